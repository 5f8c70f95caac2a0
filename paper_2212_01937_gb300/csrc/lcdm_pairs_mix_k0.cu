// Pair-kernel instantiations: precision mix, 0 tangent directions.
#include "lcdm_launch.cuh"
namespace lcdm {
PairsTable table_mix_k0() { return value_table<1>(); }
}
