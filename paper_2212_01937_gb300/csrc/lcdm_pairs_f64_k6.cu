// Pair-kernel instantiations: precision f64, 6 tangent directions.
#include "lcdm_launch.cuh"
namespace lcdm {
PairsTable table_f64_k6() { return tangent_table<0, 6>(); }
}
