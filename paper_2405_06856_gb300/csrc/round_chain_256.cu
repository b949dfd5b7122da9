// The placement chain of tables of up to 256 slots.
#include "round_chain.cuh"

namespace aladdin {
template cudaError_t round_chain_e<8>(const DevParams&, const ClusterDev&, const RoundIO&,
                                       const RoundChainBuffers*, cudaStream_t, bool*);
template bool chain_serves_sim_e<8>(int, int, int, int);
}  // namespace aladdin
