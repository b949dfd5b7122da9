// The placement chain of tables of up to 1024 slots.
#include "round_chain.cuh"

namespace aladdin {
template cudaError_t round_chain_e<32>(const DevParams&, const ClusterDev&, const RoundIO&,
                                       const RoundChainBuffers*, cudaStream_t, bool*);
template bool chain_serves_sim_e<32>(int, int, int, int);
}  // namespace aladdin
