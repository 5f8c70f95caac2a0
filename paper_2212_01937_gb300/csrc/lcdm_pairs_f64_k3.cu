// Pair-kernel instantiations: precision f64, 3 tangent directions.
#include "lcdm_launch.cuh"
namespace lcdm {
PairsTable table_f64_k3() { return tangent_table<0, 3>(); }
}
