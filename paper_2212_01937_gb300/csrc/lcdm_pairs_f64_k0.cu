// Pair-kernel instantiations: precision f64, 0 tangent directions.
#include "lcdm_launch.cuh"
namespace lcdm {
PairsTable table_f64_k0() { return value_table<0>(); }
}
