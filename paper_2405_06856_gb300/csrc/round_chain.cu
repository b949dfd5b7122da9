// K4 as a chain: which instantiation of round_chain.cuh (one translation unit
// each, for the build's sake) serves a round.
#include <algorithm>

#include "aladdin_host.h"

namespace aladdin {

template <int E>
cudaError_t round_chain_e(const DevParams& P, const ClusterDev& C, const RoundIO& io,
                          const RoundChainBuffers* B, cudaStream_t st, bool* used);
template <int E>
bool chain_serves_sim_e(int W, int cap, int K, int smem_max);

constexpr size_t CH_FLAGS_MAX = (size_t)512 << 20;  // bytes of rank-order flags a chunk holds

// Workers below which a direct round evaluates workers as it goes instead of
// scoring every pair first.
constexpr int CH_FLAGS_MIN_W = 192;

static bool ch_flags(const ClusterDev& C, const RoundIO& io)
{
    return C.W >= CH_FLAGS_MIN_W && io.n_cand >= 64;
}

size_t round_chain_flag_bytes(const DevParams& P, const ClusterDev& C, const RoundIO& io)
{
    if (io.sim || P.groups > 1 || !ch_flags(C, io)) return 0;
    const size_t ldf = (size_t)((C.W + 31) & ~31);
    const size_t chunk = std::min<size_t>((size_t)io.n_cand, std::max<size_t>(1, CH_FLAGS_MAX / ldf));
    return chunk * ldf;
}

bool round_chain_serves_sim(int W, int cap, int K)
{
    DevInfo d;
    if (device_info(&d) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    switch (lanes_per_worker(cap)) {
    case 1:
    case 2:
    case 4: return chain_serves_sim_e<4>(W, cap, K, d.smem_optin);
    case 8: return chain_serves_sim_e<8>(W, cap, K, d.smem_optin);
    case 16: return chain_serves_sim_e<16>(W, cap, K, d.smem_optin);
    case 32: return chain_serves_sim_e<32>(W, cap, K, d.smem_optin);
    default: return false;
    }
}

cudaError_t launch_round_chain(const DevParams& P, const ClusterDev& C, const RoundIO& io,
                               const RoundChainBuffers* B, cudaStream_t st, bool* used)
{
    *used = false;
    if (P.wait_test || (!io.sim && io.n_cand <= 0) || (!io.sim && !B)) return cudaSuccess;
    switch (lanes_per_worker(C.cap)) {
    case 1:
    case 2:
    case 4: return round_chain_e<4>(P, C, io, B, st, used);
    case 8: return round_chain_e<8>(P, C, io, B, st, used);
    case 16: return round_chain_e<16>(P, C, io, B, st, used);
    case 32: return round_chain_e<32>(P, C, io, B, st, used);
    default: return cudaSuccess;
    }
}

}  // namespace aladdin
