// Pair-kernel instantiations: precision f64, 4 tangent directions.
#include "lcdm_launch.cuh"
namespace lcdm {
PairsTable table_f64_k4() { return tangent_table<0, 4>(); }
}
