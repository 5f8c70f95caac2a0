// Pair-kernel instantiations: precision mix, 4 tangent directions.
#include "lcdm_launch.cuh"
namespace lcdm {
PairsTable table_mix_k4() { return tangent_table<1, 4>(); }
}
