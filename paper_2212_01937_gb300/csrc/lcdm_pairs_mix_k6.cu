// Pair-kernel instantiations: precision mix, 6 tangent directions.
#include "lcdm_launch.cuh"
namespace lcdm {
PairsTable table_mix_k6() { return tangent_table<1, 6>(); }
}
