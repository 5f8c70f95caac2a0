// Pair-kernel instantiations: precision mix, 3 tangent directions.
#include "lcdm_launch.cuh"
namespace lcdm {
PairsTable table_mix_k3() { return tangent_table<1, 3>(); }
}
