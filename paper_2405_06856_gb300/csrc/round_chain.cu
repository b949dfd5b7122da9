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

// Whether a direct round scores every pair first (a launch, then a look is a
// scan of one row of flags) or its look-ahead evaluates workers as it goes.
// Calls of 64 candidates, with flags / without, us: 64 workers 140 / 139 (128
// slots) and 175 / 195 (512), 128 workers 176 / 188 and 154 / 245, 512 workers
// 189 / 271 and 188 / 852; of 16 candidates: 64 workers 82 / 77 and 105 / 111, 256
// workers 116 / 125 and 99 / 162. The line lies where they meet.
constexpr int CH_FLAGS_MIN_W = 64;
constexpr long long CH_FLAGS_MIN_PAIRS = 4096;

static bool ch_flags(const ClusterDev& C, const RoundIO& io)
{
    return C.W >= CH_FLAGS_MIN_W && (long long)C.W * io.n_cand >= CH_FLAGS_MIN_PAIRS;
}

int round_chain_chunk(const DevParams& P, const ClusterDev& C, const RoundIO& io)
{
    if (io.sim || P.groups > 1 || P.wait_test || !ch_flags(C, io)) return 0;
    const size_t rows = std::max<size_t>(1, CH_FLAGS_MAX / (size_t)round_flag_row(C.W));
    return (int)std::min<size_t>((size_t)io.n_cand, rows);
}

// Workers up to which a simulation's rounds run as a chain: its looks evaluate 32
// workers at a time, so past a line the sliced round is faster. Alone it spans
// several CTAs; beside others (the probes of a search) it has one. Steady
// traces, sliced round / chain: 32 slots 0.94 at 32 workers and 0.88 at 96; 64
// slots 0.95 and 0.93; 128 slots 1.09 at 96, 0.99-1.07 at 192, 0.90-1.03 at 256; 256
// slots 1.05-1.18 at 192, 0.94-1.12 at 256; 512 slots 1.01-1.26 at 448, 0.72-0.96
// at 512; 1,024 slots 0.99-1.23 at 384, 0.72-0.94 at 448.
static int ch_sim_line(int cap, bool beside)
{
    switch (lanes_per_worker(cap)) {
    case 1: return beside ? 96 : 0;
    case 2: return beside ? 128 : 0;
    case 4: return beside ? 256 : 192;
    case 8: return beside ? 320 : 224;
    case 16: return 448;
    default: return 384;
    }
}

bool round_chain_serves_sim(int W, int cap, int K, bool beside)
{
    if (W > ch_sim_line(cap, beside)) return false;
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
    if (io.sim && C.W > ch_sim_line(C.cap, io.single_cta != 0)) return cudaSuccess;
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
