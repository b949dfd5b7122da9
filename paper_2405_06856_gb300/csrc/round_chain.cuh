// K4: one greedy best-fit placement round (Algorithm 1) as a chain of exact
// single-pair decisions.
//
// Candidates are placed in index order and each one sees the state the earlier
// ones left, so a round is a sequential chain and its time is the latency of
// one link times the candidates. Committing a candidate to worker i only adds
// a request to i: every other worker keeps its state, its table and its
// capacity_norm. And most candidates go to a worker that took one of the last
// few (best fit fills the fullest worker that still takes the request; two to
// eight workers receive 90-98% of a round). So the chain keeps two of the
// last winners "hot": their requests sit in the registers of four warps each,
// with the exact integer aggregates of the projection at each request's
// last iteration (iterations and context tokens run until then, KV held at
// it). For a hot worker
//   * a candidate's test needs no table: each request tests the candidate's
//     prompt against its own bound, and one vote ends the pair. The bounds are
//     the table's (same functions, same roundings); the minima the table
//     stores are only ever compared, so testing every request gives the same
//     answer;
//   * an appended request changes each aggregate by a term of its own, so
//     nothing is sorted or scanned: a link updates the aggregates, re-forms
//     the bounds and tests the next candidate.
// Of the CTA's 16 warps eight hold the hot workers; one decides each link from
// their votes and the look-ahead's record; one forms the hot workers' own terms
// (KV at the candidate's end, TTFT, the candidate's own decode bound); six look
// ahead: for each of the next candidates they find its best choice among the
// workers that are not hot (the first feasible worker the round has not
// modified, in the round-start capacity_norm order, and the feasible modified
// worker of largest key). Only when that record wins (a "miss") does a worker
// change places: the hot worker used least recently leaves, its table formed
// from its aggregates (the bits that a table build forms, without its sorts and
// sums), while look-ahead warps load and sum the new worker's requests (its
// sorted keys are kept by every table build) and look at the next candidates
// among the others.
//
// Bound: the link's latency, a chain of dependent register arithmetic, a vote,
// two barriers and a reduction at 45% of the SM's issue slots. On tables of up
// to 128 and 512 slots a plain link takes 1,150 and 1,300 cycles and a miss 7,000
// and 11,000. Measured against rebuilding the winner's table at every link: 2,048
// candidates on 256 workers 5.3 -> 1.70 ms, 13,107 on 16,384 workers (1,024
// slots) 84 -> 17 ms, 31 groups on 4,096 workers 2.75 -> 0.87 ms, a simulation
// of 128 workers 37.2 -> 23.4 ms. A round whose candidates spread over ever other
// workers is all misses: on tables of 32 slots it is 0.7 to 0.9 times as fast as
// rebuilding them (875 candidates on 14,000 workers 4.8 -> 5.9 ms), on larger ones
// 0.85 to 1.3.
//
// Where the round has a candidate x worker flag matrix (direct rounds of
// larger fleets, scored by the scoring kernel against the round-start state in
// rank order), the first feasible unmodified worker is a scan of one row;
// otherwise the look-ahead warps evaluate the workers in rank order, 32 at a
// time, until one takes the candidate.
//
// Direct mode places the caller's candidates; grouped scheduling in direct
// mode runs one CTA per group on the group's candidates and workers (they
// share nothing); trace mode (fleet simulation) places the waiting requests
// and the heartbeat's arrivals as k_round does.
#pragma once

#include <algorithm>

#include "round_common.cuh"

// A lambda over register state has to be part of its caller: a call would put
// everything that it captures into memory.
#define CH_INLINE __attribute__((always_inline))

namespace aladdin {

constexpr int CH_THREADS = 512;
constexpr int CH_WARPS = CH_THREADS / 32;
constexpr int CH_HOT = 8;                     // warps holding hot workers
constexpr int CH_DECIDE = CH_HOT;             // the warp that decides a link
constexpr int CH_TERMS = CH_HOT + 1;          // the warp that forms the workers' own terms
constexpr int CH_LOOK0 = CH_HOT + 2;          // first warp looking ahead
constexpr int CH_SCAN = CH_WARPS - CH_LOOK0;  // warps looking ahead
constexpr int CH_RING = 64;                   // candidate records in shared memory
// Candidates looked ahead at a time: a miss ends looks that are under way, and
// looks slow the links beside them. 30, 18 and 12 took a round of 256 workers 1.82, 1.67
// and 1.68 ms, a simulation of 128 workers 25.2, 24.0 and 23.6 ms, 31 groups on 4,096
// workers 0.96, 0.90 and 0.87 ms.
constexpr int CH_AHEAD = 12;
// Candidates looked at during a change of the hot worker in a simulation, where
// most candidates change it: by the look-ahead warps that do not stage the new
// one (elsewhere every look-ahead warp takes one).
constexpr int CH_FIRST = 2;
// Rows of 512 flags that a look has in flight past the first.
constexpr int CH_ROWS = 4;
constexpr int CH_WIN = 1024;                  // rank positions kept in shared memory
constexpr int CH_SORT_MAX = 512;              // workers a trace-mode round ranks by itself
constexpr int CH_MAX_SLOTS = 4096;            // modified workers held, at most
constexpr int CH_RC_MAX = 64;                 // breakpoint samples of one in shared memory, at most
constexpr int CH_TSHIFT = 2;                  // without flags: every 4th breakpoint is sampled
constexpr int CH_TS_MAX = 64;                 // samples of one, at most
// A round with flags starts afresh (the rest of the candidates scored against the
// state so far) when it has modified this many workers: every look holds its
// candidate against each of them. 6,000 candidates on 6,000 workers of 32 slots:
// 46.7 ms without, 28.5, 24.6 and 23.0 at 768, 384 and 192; 13,107 on 16,384 (which
// modify 204) 16.76, and 17.04 at 192.
constexpr int CH_FRESH = 256;
constexpr int CH_TRIAL = 48;                  // candidates before a group's chain is compared
constexpr int CH_UB = 32;                     // prompt limits of one, by predicted length
constexpr int CH_KV_MAX = 1 << 29;            // KV usage saturates here (M < 2^24)
constexpr int CH_HJ_MAX = 1 << 25;            // h and j likewise: one token would exceed M

// Tables of up to 128 slots share E = 4. A hot worker's requests: EPL a lane
// over NWG warps; KH hot workers. (1,024 slots over four warps, eight requests a
// lane, spilled a kilobyte of registers: a change of the hot worker took 28,000
// cycles, a round of 13,107 candidates 17.9 ms against 17.1.)
template <int E>
struct ChCfg {
    static constexpr int NWG = E >= 32 ? 8 : 4;
    static constexpr int EPL = E / NWG;
    static constexpr int KH = CH_HOT / NWG;
    // Look-ahead warps that load (stage) the next hot worker, their elements a
    // lane, and the requests that they hold. On 1,024-slot tables, whose eight hot
    // warps load a small worker themselves in little time, they do so in direct
    // rounds up to 128 requests (the look-ahead warps have six candidates to look
    // at then); a simulation stages all that fit (147 workers of about 90 requests
    // 1.29 ms a heartbeat against 1.50).
    static constexpr int LN = 4, LE = EPL, LCAP = 32 * LN * LE;
    static __device__ __forceinline__ bool staged(int n, bool sim)
    {
        return NWG == LN || (n < LCAP && (sim || n > 128));
    }
};

// Round-start entry of a rank position: the worker there, its key and count.
struct __align__(16) RankEnt {
    unsigned long long key;
    int w;
    int n;
};

struct ChArgs {
    DevParams P;
    ClusterDev C;
    RoundIO io;
    const uint8_t* F;    // [n_cand][ldf] flags of the round-start state, rank order, or nullptr
    int ldf;             // row stride of F (a multiple of 32)
    RankEnt* rank_ent;   // [W] scratch of rank positions beyond the ones in shared memory
    int* c_stop;         // out (direct, of each group): first candidate left to another kernel
    int placed_cost, other_cost;  // groups: cycles that k_round_grp takes for a candidate
                                  // that is placed and for another (0: not compared)
    int* votes;          // groups whose chain is the slower way
    int mmax;            // modified workers held
    int rc;              // breakpoint samples of one in shared memory
    int nub;             // prompt limits of one (CH_UB + 1, or 0: none)
    int nts;             // without F: breakpoint samples of every worker, by rank position
    int nwin;            // rank positions in shared memory
};

struct ChSums {          // over a worker's requests, split at a remaining length r
    int n, A;            // requests longer than r, their context
    int PR;              // remaining iterations of the others
    int pad;
    long long PRA;       // sum of r_j a_j + r_j (r_j + 1) / 2 of the others
};

// A request's aggregates at its own last iteration.
struct __align__(16) ChElem {
    long long SK;        // context tokens summed over iterations 1..r
    int Sb;              // requests summed over them
    int kv;              // KV usage at iteration r (saturated)
};

// A hot worker's own terms.
struct ChOwn {
    int w, m;            // worker, slot
    int n, M, sumP, npend, sumIn, sumPred;
    float s, inv_s, off, wpmax;
    double dmin;
};

// What ended a run of links (negative decisions after CH_NOBODY end it).
constexpr int CH_DONE = 0, CH_MISS = 1, CH_STOP = 2;
constexpr int CH_NOBODY = -1, CH_END = -2;

template <int E>
struct ChSmem {
    using Cfg = ChCfg<E>;
    CandRec rec[CH_RING];            // by candidate index mod CH_RING
    int4 raw[CH_RING];               // prompt, predicted, real output length, group
    double wd[CH_RING];              // wait (ms)
    long long tix[CH_RING];          // trace mode: trace index
    float4 rc[CH_RING];              // wait, theta T_dec r, shared_time(r), -
    unsigned short frow[CH_RING][32];  // feasible bits of rank positions 0..511
    unsigned long long alt_k[CH_RING];  // best choice among the workers not hot
    int alt_w[CH_RING], alt_f[CH_RING];
    int alt_at[CH_RING];             // 1 + the candidate it was looked at for, or 0
    int lw_[CH_RING], ln[CH_RING];   // log: each candidate's worker (-1, -2) and slot
    // by candidate parity, double-buffered
    ChSums ps[2][CH_HOT];            // each hot warp's partial sums
    unsigned vote[2][CH_HOT];        // its requests admit the candidate
    unsigned own_ok[2][Cfg::KH][2];  // the worker's own terms do [previous one appended or not]
    ChElem ne[2][Cfg::KH][2];        // the candidate's aggregates, were it appended [same]
    int dec[2];                      // its hot slot, CH_NOBODY or CH_END
    ChSums ld[32];                   // load: chunk totals (n unused; A, PR, PRA inclusive)
    int ls[CH_HOT][4];               // load: sum in (pending), sum in, sum pred, pending
    float lw[CH_HOT];                // load: largest wait
    double lm[CH_HOT];               // load: smallest saved decode time
    ChOwn own[Cfg::KH];              // as of the latest load
    int hw[CH_HOT], hm[CH_HOT];      // hot workers and their slots when a run ends
    int hn[CH_HOT];                  // their requests when they were loaded
    // a leaving worker's requests: keys (r << 10 | slot) before and after
    // sorting, and the rest in sorted order
    alignas(16) unsigned nkey[32 * E + 4];
    unsigned okey[32 * E], key[32 * E];
    int ea[32 * E], ekv[32 * E], eSb[32 * E];
    long long eSK[32 * E];
    float ebnd[32 * E], esg[32 * E];
    // a worker that becomes hot, formed by look-ahead warps while the hot ones
    // write the leaving worker's table (bit 31 of sta: placed in this round)
    static constexpr int ST = Cfg::LCAP;
    int str[ST], sta[ST], stS[ST], stk[ST];
    long long stK[ST];
    float stb[ST], sty[ST], std_[ST];
    ChOwn sto;
    int ti[4][32];                   // a leaving worker's chunks' totals: rows, KV peaks, context
    float tf[4][32];                 // and bounds
    int code[2], next[2];            // [run parity]
    int slow[2];                     // the rest is left to k_round_grp [same]
    int miss_w, miss_f, victim;
    int miss_n;                      // the new hot worker's requests
    int left_n;                      // requests of the worker that left last
    int abort, never;                // a run has ended; always 0
    int cnt[CH_WARPS + 1];
    int lq[CH_SCAN][64];             // look-ahead: slots to evaluate
};

constexpr int CH_FULL = 1 << 29;   // winner flags: the worker has no free slot
constexpr int CH_UNMOD = 1 << 28;  // not modified yet (low bits: its rank position, else its slot)
constexpr int CH_IDX = (1 << 28) - 1;

// Bit b of the result: flag byte b of the 16 is 15 (feasible).
__device__ __forceinline__ unsigned feasible16(const uint4 u)
{
    const unsigned w[4] = {u.x, u.y, u.z, u.w};
    unsigned bits = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        // equal bytes -> their low bits gathered into a nibble by a multiply
        // (no two partial products overlap)
        const unsigned eq = __vcmpeq4(w[i], 0x0f0f0f0fu) & 0x01010101u;
        bits |= ((eq * 0x10204080u) >> 28) << (4 * i);
    }
    return bits;
}

__device__ __forceinline__ void cta_sync() { asm volatile("bar.sync 0;" ::: "memory"); }

// The hot warps of one slot (one slot loads at a time).
template <int N>
__device__ __forceinline__ void hot_group_sync()
{
    asm volatile("bar.sync 4, %0;" ::"r"(N * 32) : "memory");
}

// The warps looking ahead, among themselves.
__device__ __forceinline__ void look_sync()
{
    asm volatile("bar.sync 2, %0;" ::"n"(CH_SCAN * 32) : "memory");
}

// The warps that stage a worker among themselves, and its handing over.
template <int N>
__device__ __forceinline__ void stage_group_sync()
{
    asm volatile("bar.sync 6, %0;" ::"r"(N * 32) : "memory");
}
template <int N>
__device__ __forceinline__ void staged_arrive()
{
    asm volatile("bar.arrive 7, %0;" ::"r"(N * 32) : "memory");
}
template <int N>
__device__ __forceinline__ void staged_wait()
{
    asm volatile("bar.sync 7, %0;" ::"r"(N * 32) : "memory");
}

// A link's two barriers: votes and terms are in (hot warps, CH_DECIDE and
// CH_TERMS), and the decision is out (CH_DECIDE arrives, the hot warps wait).
__device__ __forceinline__ void votes_sync()
{
    asm volatile("bar.sync 3, %0;" ::"r"((CH_HOT + 2) * 32) : "memory");
}
__device__ __forceinline__ void decision_wait()
{
    asm volatile("bar.sync 5, %0;" ::"r"((CH_HOT + 1) * 32) : "memory");
}
__device__ __forceinline__ void decision_arrive()
{
    asm volatile("bar.arrive 5, %0;" ::"r"((CH_HOT + 1) * 32) : "memory");
}

// A hot worker's requests in the registers of its warps. Elements past the
// last request are neutral: r = 0 (they count as finished before any
// candidate), kv lowest, num +inf.
template <int EPL>
struct Hot {
    int r[EPL], a[EPL];
    int Sb[EPL], kv[EPL];  // ChElem
    long long SK[EPL];
    float num[EPL];        // prompt bound x its cost, finishing with or before the candidate
    float sg[EPL];         // slack, finishing after it
    // theta T_dec r + bank, the candidate's share of its iterations and the
    // prompt's cost (shared_time, prompt_cost_*), and h r (saturated)
    float hb[EPL], hy[EPL], hd[EPL];
    int hh[EPL];
    unsigned pend;         // bit e: placed in this round
    int n, M, sumP;
    float s, inv_s, stallk;
};

// r (r + 1) / 2 in 32 bits
__device__ __forceinline__ unsigned tri32(int r) { return (unsigned)((r + 1) >> 1) * (unsigned)(r | 1); }

template <int V>
struct IntC {
    static constexpr int value = V;
};

template <int E>
__global__ void __launch_bounds__(CH_THREADS, 1) k_round_chain(ChArgs A)
{
    using Cfg = ChCfg<E>;
    constexpr int NWG = Cfg::NWG, EPL = Cfg::EPL, KH = Cfg::KH;
    static_assert(NWG * EPL == E && EPL <= 4, "the capacity is covered, in registers");
    extern __shared__ __align__(16) unsigned char smraw[];
    ChSmem<E>& sm = *reinterpret_cast<ChSmem<E>*>(smraw);
    const DevParams& P = A.P;
    const ClusterDev& C = A.C;
    const RoundIO& io = A.io;
    const int mmax = A.mmax, rc = A.rc, nwin = A.nwin, nub = A.nub, nts = A.nts;
    const int rs = rc + R2_RHO_PAD;  // a slot's stride: an odd number of words
    unsigned char* tail = smraw + ((sizeof(ChSmem<E>) + 15) / 16) * 16;
    RankEnt* win = reinterpret_cast<RankEnt*>(tail);
    float4* mwrec = reinterpret_cast<float4*>(win + nwin);
    unsigned long long* mkey = reinterpret_cast<unsigned long long*>(mwrec + mmax);
    int* mw = reinterpret_cast<int*>(mkey + mmax);
    int* mR = mw + mmax;
    int* mn = mR + mmax;   // requests; bit 31: hot (its table is not current)
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int cap = C.cap;
    const bool sim = io.sim != 0;

    // This CTA's candidates (local index i is candidate c0 + i G) and workers.
    const int GP = P.groups;                       // scheduling groups
    const int G = sim ? 1 : (GP > 1 ? GP : 1);     // chains: one CTA a group in direct mode
    const int g = blockIdx.x;
    const bool filter = sim && GP > 1;             // trace mode: one chain, workers filtered
    int c0 = 0, n_wait0 = 0, n_cand;
    if (sim) {
        if (*io.status != 0) return;
        n_wait0 = *io.n_wait;
        n_cand = n_wait0 + (int)(io.arr_end - io.arr_begin);
    } else {
        c0 = G > 1 ? (int)((((long long)g - io.rid0 % G) % G + G) % G) : 0;
        n_cand = c0 < io.n_cand ? (io.n_cand - c0 + G - 1) / G : 0;
    }
    const int W = G > 1 ? (C.W > g ? (C.W - g + G - 1) / G : 0) : C.W;  // workers of this chain
    RankEnt* const rank_ent =
        A.rank_ent + (G > 1 ? (long long)g * (C.W / G) + min(g, C.W % G) : 0);
    const int nwords = (W + 31) >> 5;
    unsigned* modbits = reinterpret_cast<unsigned*>(mn + mmax);
    float* mub = reinterpret_cast<float*>(modbits + ((nwords + 3) & ~3));  // [mmax][nub]
    unsigned short* rho = reinterpret_cast<unsigned short*>(mub + (size_t)mmax * nub);
    int shift = 0;  // every (1 << shift)-th breakpoint is sampled
    while ((cap >> shift) > CH_RC_MAX) ++shift;
    // every worker's samples (nts of them, tail of shared memory): the first
    // ones stand in for the whole table where a worker holds few requests
    unsigned short* const trho = rho + (size_t)mmax * rs;
    const int ts = nts + R2_RHO_PAD;
    const int tshift = CH_TSHIFT;

    // the round-start rank order of this chain's workers
    if (n_cand > 0) {
        auto put = [&](int p, int w) {
            RankEnt e;
            e.key = C.key[w];
            e.w = w;
            e.n = C.n[w];
            if (p < nwin) win[p] = e;
            else rank_ent[p] = e;
        };
        if (sim) {
            // W <= nwin: a bitonic sort of (key, index) in shared memory
            int m = 1;
            while (m < W) m <<= 1;
            for (int p = tid; p < m; p += CH_THREADS) {
                if (p < W) put(p, p);
                else win[p] = RankEnt{0ull, p, 0};  // padding sorts last
            }
            __syncthreads();
            for (int size = 2; size <= m; size <<= 1) {
                for (int st = size >> 1; st > 0; st >>= 1) {
                    for (int t = tid; t < m / 2; t += CH_THREADS) {
                        const int i = ((t & ~(st - 1)) << 1) | (t & (st - 1));
                        const RankEnt x = win[i], y = win[i + st];
                        const bool y_first = y.key > x.key || (y.key == x.key && y.w < x.w);
                        if (y_first == ((i & size) == 0)) {
                            win[i] = y;
                            win[i + st] = x;
                        }
                    }
                    __syncthreads();
                }
            }
        } else if (G == 1) {
            for (int p = tid; p < W; p += CH_THREADS) put(p, C.order[p]);
        } else {
            // the group's workers in the order of the whole cluster's
            const int per = (C.W + CH_THREADS - 1) / CH_THREADS;
            const int p0 = min(C.W, tid * per), p1 = min(C.W, p0 + per);
            int cnt = 0;
            for (int p = p0; p < p1; ++p) cnt += C.order[p] % G == g;
            int incl = cnt;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int u = __shfl_up_sync(FULL, incl, d);
                if (lane >= d) incl += u;
            }
            if (lane == 31) sm.cnt[warp] = incl;
            __syncthreads();
            int at = incl - cnt;
            for (int k = 0; k < warp; ++k) at += sm.cnt[k];
            for (int p = p0; p < p1; ++p) {
                const int w = C.order[p];
                if (w % G == g) put(at++, w);
            }
        }
    }
    for (int k = tid; k < nwords; k += CH_THREADS) modbits[k] = 0u;
    if (nts > 0 && n_cand > 0) {
        __syncthreads();  // the rank order
        for (int k = tid; k < W * nts; k += CH_THREADS) {
            const int p = k / nts, i = k - p * nts;
            const int w = p < nwin ? win[p].w : rank_ent[p].w, row = ((i + 1) << tshift) - 1;
            if (row < C.R[w])
                trho[p * ts + i] = (unsigned short)(
                    __float_as_int(C.tab[((long long)w * C.rows + row) * ROW_F4].x) - 1);
        }
    }

    auto fetch = [&](int k) CH_INLINE {
        const int b = k & (CH_RING - 1);
        int32_t a, r, rl;
        double wd;
        long long id = k;
        if (sim) {
            id = k < n_wait0 ? io.wl[k] : io.arr_begin + (k - n_wait0);
            a = io.tin[id];
            r = io.tpred[id];
            rl = io.treal ? io.treal[id] : r;
            wd = io.t_now - io.t_arr[id];
        } else {
            const int c = c0 + k * G;
            a = io.in[c];
            r = io.pred[c];
            rl = r;
            wd = io.wait ? (double)io.wait[c] : 0.0;
        }
        const CandRec cq = make_cand(P, a, r, (float)wd, k);
        sm.rec[b] = cq;
        sm.raw[b] = make_int4(a, r, rl, filter ? (int)(id % GP) : 0);
        sm.wd[b] = wd;
        sm.rc[b] = make_float4((float)wd, slack_base(P, cq.r, 0.0f), shared_time(P, cq.r), 0.0f);
        sm.tix[b] = id;
    };
    // a look-ahead warp: candidate k's first flags, kept until it is looked at
    auto fetch_row = [&](int k) CH_INLINE {
        unsigned bits = 0;
        if (16 * lane < W) bits = feasible16(__ldg(reinterpret_cast<const uint4*>(A.F + (size_t)k * A.ldf) + lane));
        sm.frow[k & (CH_RING - 1)][lane] = (unsigned short)bits;
    };
    int rec_end = min(n_cand, 2 * CH_AHEAD);  // candidates fetched
    if (warp == CH_WARPS - 1)
        for (int k = lane; k < rec_end; k += 32) fetch(k);
    if (A.F && warp >= CH_LOOK0)
        for (int k = warp - CH_LOOK0; k < rec_end; k += CH_SCAN) fetch_row(k);
    if (tid == 0) sm.abort = sm.never = 0;
    if (tid < CH_RING) sm.alt_at[tid] = 0;
    __syncthreads();

    int mcount = 0;  // modified workers (every thread tracks the same value)
    int c = 0;       // the next candidate

    // Table row of length r (rb: the worker's rows, R breakpoints) from n
    // samples of every (1 << sh)-th one: they bound it to one stretch, searched
    // in the table.
    auto find_sampled = [&](const unsigned short* sp, int n, int sh, long long rb, int R,
                            int r) CH_INLINE {
        const int m = min(R >> sh, n);
        int lo = 0, hi = m;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if ((int)sp[mid] >= r) hi = mid;
            else lo = mid + 1;
        }
        const bool last = lo == m;  // past the last sample
        lo <<= sh;
        hi = last ? R : lo + (1 << sh) - 1;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (__float_as_int(C.tab[(rb + mid) * ROW_F4].x) > r) hi = mid;
            else lo = mid + 1;
        }
        return lo;
    };
    auto slot_row = [&](int i, long long rb, int R, int r) CH_INLINE {  // a modified worker's
        return find_sampled(rho + (long long)i * rs, rc, shift, rb, R, r);
    };
    // Lengths r by half octaves: the limit's index and the smallest r in it.
    auto ub_index = [](int r) {
        const int l = 31 - __clz(r);
        return min(CH_UB - 1, 2 * l + (l > 0 ? (r >> (l - 1)) & 1 : 0));
    };
    auto ub_least = [](int i) { return (1 << (i >> 1)) + ((i & 1) ? (1 << (i >> 1)) >> 1 : 0); };

    // A look-ahead warp: candidate k's best choice among the workers that are
    // not hot.
    auto look = [&](int k, const int* stop) CH_INLINE {
        auto stopped = [&]() { return __any_sync(FULL, *(const volatile int*)stop) != 0; };
        const int b = k & (CH_RING - 1);
        const CandRec cq = sm.rec[b];
        unsigned long long bk = 0ull;
        int bw = NONE, bf = 0;
        if (cq.valid) {
            const int grp = filter ? sm.raw[b].w : 0;
            if (A.F) {
                // 512 positions first (most candidates end there), then 2,048 at a
                // time: the row's loads are what a long scan waits for
                const uint8_t* row = A.F + (size_t)k * A.ldf;
                int pos = -1;
                auto open = [&](unsigned bits, int p0) CH_INLINE {  // the first one open from p0 on
                    if (p0 < W) bits &= ~(modbits[p0 >> 5] >> (p0 & 16)) & 0xffffu;
                    if (W - p0 < 16) bits &= W > p0 ? (1u << (W - p0)) - 1u : 0u;
                    const unsigned who = __ballot_sync(FULL, bits != 0);
                    if (who) pos = __shfl_sync(FULL, p0 + __ffs(bits) - 1, __ffs(who) - 1);
                };
                open(sm.frow[b][lane], 16 * lane);
                for (int base = 512; base < W && pos < 0; base += 512 * CH_ROWS) {
                    if (stopped()) return;
                    uint4 u[CH_ROWS];
#pragma unroll
                    for (int j = 0; j < CH_ROWS; ++j) {
                        const int p0 = base + 512 * j + 16 * lane;
                        u[j] = p0 < W ? __ldg(reinterpret_cast<const uint4*>(row + p0)) : uint4{0, 0, 0, 0};
                    }
#pragma unroll
                    for (int j = 0; j < CH_ROWS; ++j)
                        if (pos < 0) open(feasible16(u[j]), base + 512 * j + 16 * lane);
                }
                if (pos >= 0) {
                    const RankEnt e = pos < nwin ? win[pos] : rank_ent[pos];
                    bk = e.key;
                    bw = e.w;
                    bf = pos | CH_UNMOD | (e.n >= cap ? CH_FULL : 0);
                }
            } else {
                for (int base = 0; base < W; base += 32) {
                    if (stopped()) return;
                    const int pos = base + lane;
                    bool ok = false;
                    RankEnt e{0ull, 0, 0};
                    if (pos < W && !((modbits[base >> 5] >> lane) & 1u)) {
                        e = pos < nwin ? win[pos] : rank_ent[pos];
                        if (!filter || e.w % GP == grp) {
                            const long long rb = (long long)e.w * C.rows;
                            const int p =
                                find_sampled(trho + pos * ts, nts, tshift, rb, C.R[e.w], cq.ri);
                            const float4* t = C.tab + (rb + p) * ROW_F4;
                            float m;
                            ok = eval_pair_mode(P.approx != 0, t[0], t[1], C.tab2[rb + p],
                                                C.wrec[e.w],
                                                P.approx ? C.wapx[e.w] : make_float2(0.0f, 0.0f),
                                                cq, m) == 15u;
                        }
                    }
                    const unsigned who = __ballot_sync(FULL, ok);
                    if (who) {
                        const int src = __ffs(who) - 1;
                        bk = __shfl_sync(FULL, e.key, src);
                        bw = __shfl_sync(FULL, e.w, src);
                        const int en = __shfl_sync(FULL, e.n, src);
                        bf = (base + src) | CH_UNMOD | (en >= cap ? CH_FULL : 0);
                        break;
                    }
                }
            }
            // Modified workers whose key could beat that and whose prompt limit
            // at this length lets the candidate in (most are full): those that
            // remain are gathered, up to one a lane, and evaluated.
            const int ui = ub_index(cq.ri);
            int* const lq = sm.lq[warp - CH_LOOK0];
            int held = 0;  // slots gathered in lq (uniform)
            auto evaluate = [&](int i) {
                const int w = mw[i];
                const long long rb = (long long)w * C.rows;
                const long long row = rb + slot_row(i, rb, mR[i], cq.ri);
                const float4* t = C.tab + row * ROW_F4;
                float m;
                const unsigned f =
                    eval_pair_mode(P.approx != 0, t[0], t[1], C.tab2[row], mwrec[i],
                                   P.approx ? C.wapx[w] : make_float2(0.0f, 0.0f), cq, m);
                if (f == 15u) better_f(bk, bw, bf, mkey[i], w, i | (mn[i] >= cap ? CH_FULL : 0));
            };
            const unsigned long long uk = bk;  // the unmodified worker's, the same in every lane
            const int uw = bw;
            for (int i0 = 0; i0 < mcount; i0 += 32) {
                if ((i0 & 127) == 96 && stopped()) return;
                const int i = i0 + lane;
                bool on = i < mcount && mn[i] >= 0;  // not hot
                if (on) {
                    const unsigned long long key = mkey[i];
                    const int w = mw[i];
                    on = !(nub > 0 && cq.a > mub[i * nub + ui]) &&
                         (uw == NONE || key > uk || (key == uk && w < uw)) &&
                         (!filter || w % GP == grp);
                }
                const unsigned who = __ballot_sync(FULL, on);
                if (on) lq[held + __popc(who & ((1u << lane) - 1u))] = i;
                held += __popc(who);
                __syncwarp();
                if (held >= 32) {
                    evaluate(lq[lane]);
                    held -= 32;
                    const int rest = lane < held ? lq[32 + lane] : 0;
                    __syncwarp();
                    if (lane < held) lq[lane] = rest;
                    __syncwarp();
                }
            }
            if (lane < held) evaluate(lq[lane]);
            __syncwarp();
            reduce_f(bk, bw, bf);
        }
        if (lane == 0) {
            sm.alt_k[b] = bk;
            sm.alt_w[b] = bw;
            sm.alt_f[b] = bf;
            sm.alt_at[b] = k + 1;
        }
    };

    const int hc = min(P.h, CH_HJ_MAX), jc = min(P.j, CH_HJ_MAX);
    auto sat = [](long long x) { return x > CH_KV_MAX ? CH_KV_MAX : (int)x; };
    const bool half_gamma = P.gammad == 0.5;
    auto hot_key = [&](int n, int in, int pred) {
        if (half_gamma) {
            const unsigned b2 = 2u * (unsigned)n, s2 = 2u * (unsigned)in + (unsigned)pred;
            return (unsigned long long)b2 * b2 + (unsigned long long)s2 * s2 + 1ull;
        }
        return norm_key(P, n, in, pred);
    };
    // aggregates of a new request (prompt a, output r) on a worker whose
    // requests sum to t, split at r
    auto new_elem = [&](const ChSums& t, int a, int r) CH_INLINE {
        ChElem o;
        const unsigned tri = tri32(r);
        o.Sb = t.PR + r * t.n + r;
        o.SK = t.PRA + (long long)t.n * tri + (long long)r * t.A +
               (long long)((unsigned)r * (unsigned)a + tri);
        o.kv = sat((long long)hc * ((long long)t.A + a + (long long)r * (t.n + 1)) +
                   (long long)jc * (t.n + 1));
        return o;
    };

    // ---- hot workers: warp `warp` < CH_HOT holds part `q` of hot slot `hs` ----
    const int hs = warp / NWG, q = warp % NWG;
    auto elem = [&](int e) CH_INLINE { return (e * NWG + q) * 32 + lane; };
    // runs f with a number of elements a lane that n requests need or a little
    // more (the rest are neutral): straight-line code, so that
    // the elements' dependent steps overlap
    auto with_elems = [&](int n, auto f) CH_INLINE {
        [[maybe_unused]] constexpr int CH = 32 * NWG;
        if constexpr (EPL <= 2) {
            f(IntC<EPL>());
        } else {
            if (n <= CH) f(IntC<1>());
            else if (n <= 2 * CH) f(IntC<2>());
            else f(IntC<4>());
        }
    };
    auto set_consts = [&](Hot<EPL>& H, int e, float hb, float hy, float hd, int hh) CH_INLINE {
        H.hb[e] = hb;
        H.hy[e] = hy;
        H.hd[e] = hd;
        H.hh[e] = hh;
    };
    // this warp's share of the sums split at ri, to sm.ps[par]
    auto partial_sums = [&](const Hot<EPL>& H, int ri, int par, auto ea) CH_INLINE {
        constexpr int EA = decltype(ea)::value;
        int sn = 0, sA = 0, sR = 0;
        unsigned lo = 0, hi = 0;
#pragma unroll
        for (int e = 0; e < EA; ++e) {
            const bool gt = H.r[e] > ri;
            // r a + r (r + 1) / 2 < 2^32 (r + a <= 65536)
            const unsigned v = (unsigned)H.r[e] * (unsigned)H.a[e] + tri32(H.r[e]);
            sn += gt ? 1 : 0;
            sA += gt ? H.a[e] : 0;
            sR += gt ? 0 : H.r[e];
            lo += gt ? 0u : v & 0xffffu;
            hi += gt ? 0u : v >> 16;
        }
        sn = __reduce_add_sync(FULL, sn);
        sA = __reduce_add_sync(FULL, sA);
        sR = __reduce_add_sync(FULL, sR);
        lo = __reduce_add_sync(FULL, lo);
        hi = __reduce_add_sync(FULL, hi);
        if (lane == 0) {
            ChSums& o = sm.ps[par][warp];
            o.n = sn;
            o.A = sA;
            o.PR = sR;
            o.PRA = (long long)lo + ((long long)hi << 16);
        }
    };
    auto slot_sums = [&](int slot, int par) CH_INLINE {  // from the slot's warps' shares
        ChSums t{0, 0, 0, 0, 0};
#pragma unroll
        for (int k = 0; k < NWG; ++k) {
            const ChSums& o = sm.ps[par][slot * NWG + k];
            t.n += o.n;
            t.A += o.A;
            t.PR += o.PR;
            t.PRA += o.PRA;
        }
        return t;
    };
    // load worker w's n requests into the registers of LN warps
    auto load = [&](auto& H, ChOwn& own, int w, int n, auto ln) CH_INLINE {
        constexpr int LN = decltype(ln)::value, LE = EPL, LC = LE * LN;
        constexpr bool HOT = LN == NWG && NWG > Cfg::LN;  // by the hot warps themselves
        const int q = warp % LN;
        auto elem = [&](int e) CH_INLINE { return (e * LN + q) * 32 + lane; };
        auto group_sync = [&]() CH_INLINE {
            if constexpr (HOT) hot_group_sync<LN>();
            else stage_group_sync<LN>();
        };
        const long long base = (long long)w * cap;
        H.n = n;
        H.M = C.M[w];
        H.s = C.scale[w];
        H.inv_s = 1.0f / H.s;
        H.pend = 0;
        own.w = w;
        own.M = H.M;
        own.n = n;
        own.s = H.s;
        own.inv_s = H.inv_s;
        own.off = C.off[w];
        int sP = 0, sI = 0, sD = 0, nP = 0;
        float wp = -f_inf();
        double dm = __longlong_as_double(0x7ff0000000000000ll);
        // Sb, kv, SK first hold the inclusive prefix sums of r, a and
        // r a + r (r + 1) / 2 inside the chunk of 32
#pragma unroll
        for (int e = 0; e < LE; ++e) {
            const int x = elem(e);
            H.r[e] = H.a[e] = H.Sb[e] = H.kv[e] = 0;
            H.SK[e] = 0;
            set_consts(H, e, f_inf(), 0.0f, 0.0f, 0);
            if (e * LN * 32 >= n) continue;
            float hb = f_inf(), hy = 0.0f, hd = 0.0f;
            if (x < n) {
                const unsigned key = C.skey[base + x];
                const long long slot = base + (key & 1023u);
                const int pd = C.pend[slot], gen = C.gen[slot], pr = C.pred[slot], in = C.in[slot];
                const float bk = C.bank[slot];
                const int r = (int)(key >> 10), a = in + (pd ? 0 : gen);
                const float rf = (float)r;
                H.r[e] = r;
                H.a[e] = a;
                hb = slack_base(P, rf, pd ? 0.0f : bk);
                hy = shared_time(P, rf);
                hd = pd ? prompt_cost_new(P, H.s, rf) : prompt_cost_ongoing(P, H.s, rf);
                sI += in;
                sD += pr;
                if (pd) {
                    H.pend |= 1u << e;
                    sP += in;
                    nP += 1;
                    wp = fmaxf(wp, (float)C.wait[slot]);
                } else if (P.approx) {
                    dm = fmin(dm, saved_time(P, gen, C.tdec[slot]));
                }
            }
            set_consts(H, e, hb, hy, hd, sat((long long)hc * H.r[e]));
            H.Sb[e] = H.r[e];
            H.kv[e] = H.a[e];
            H.SK[e] = (long long)((unsigned)H.r[e] * (unsigned)H.a[e] + tri32(H.r[e]));
        }
#pragma unroll
        for (int e = 0; e < LE; ++e) {
            if (e * LN * 32 >= n) break;  // uniform
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int ur = __shfl_up_sync(FULL, H.Sb[e], d), ua = __shfl_up_sync(FULL, H.kv[e], d);
                const long long ux = __shfl_up_sync(FULL, H.SK[e], d);
                if (lane >= d) {
                    H.Sb[e] += ur;
                    H.kv[e] += ua;
                    H.SK[e] += ux;
                }
            }
        }
        sP = __reduce_add_sync(FULL, sP);
        sI = __reduce_add_sync(FULL, sI);
        sD = __reduce_add_sync(FULL, sD);
        nP = __reduce_add_sync(FULL, nP);
        wp = warp_reduce(wp, OpMax<float>());
        if (P.approx) dm = warp_reduce(dm, OpMin<double>());
        if (lane == 31) {  // chunk totals (chunks past the last request: zero)
#pragma unroll
            for (int e = 0; e < LE; ++e) {
                ChSums& o = sm.ld[e * LN + q];
                o.A = H.kv[e];
                o.PR = H.Sb[e];
                o.PRA = H.SK[e];
            }
        }
        if (lane == 0) {
            sm.ls[q][0] = sP;
            sm.ls[q][1] = sI;
            sm.ls[q][2] = sD;
            sm.ls[q][3] = nP;
            sm.lw[q] = wp;
            sm.lm[q] = dm;
        }
        group_sync();
        // chunk offsets: a scan of the E chunk totals over the lanes
        int tA = lane < LC ? sm.ld[lane].A : 0, tR = lane < LC ? sm.ld[lane].PR : 0;
        long long tX = lane < LC ? sm.ld[lane].PRA : 0;
#pragma unroll
        for (int d = 1; d < LC; d <<= 1) {
            const int ur = __shfl_up_sync(FULL, tR, d), ua = __shfl_up_sync(FULL, tA, d);
            const long long ux = __shfl_up_sync(FULL, tX, d);
            if (lane >= d) {
                tR += ur;
                tA += ua;
                tX += ux;
            }
        }
        const int allA = __shfl_sync(FULL, tA, LC - 1);
        own.sumP = own.sumIn = own.sumPred = own.npend = 0;
        own.wpmax = -f_inf();
        own.dmin = __longlong_as_double(0x7ff0000000000000ll);
#pragma unroll
        for (int k = 0; k < LN; ++k) {
            own.sumP += sm.ls[k][0];
            own.sumIn += sm.ls[k][1];
            own.sumPred += sm.ls[k][2];
            own.npend += sm.ls[k][3];
            own.wpmax = fmaxf(own.wpmax, sm.lw[k]);
            own.dmin = fmin(own.dmin, sm.lm[k]);
        }
        H.sumP = own.sumP;
#pragma unroll
        for (int e = 0; e < LE; ++e) {
            H.num[e] = H.sg[e] = f_inf();
            if (e * LN * 32 >= n) {
                H.kv[e] = -CH_KV_MAX;
                continue;
            }
            const int ch = e * LN + q;
            // (inclusive offset of the chunk before)
            const int oR = __shfl_sync(FULL, tR, ch > 0 ? ch - 1 : 0);
            const int oA = __shfl_sync(FULL, tA, ch > 0 ? ch - 1 : 0);
            const long long oX = __shfl_sync(FULL, tX, ch > 0 ? ch - 1 : 0);
            const int x = elem(e);
            const int r = H.r[e], a = H.a[e];
            const int pr = H.Sb[e] + (ch > 0 ? oR : 0), pa = H.kv[e] + (ch > 0 ? oA : 0);
            const long long px = H.SK[e] + (ch > 0 ? oX : 0);
            const int np = n - (x + 1), Ag = allA - pa;
            const bool on = x < n;
            H.Sb[e] = on ? pr + r * np : 0;
            H.SK[e] = on ? px + (long long)np * tri32(r) + (long long)r * Ag : 0;
            H.kv[e] = on ? sat((long long)hc * ((long long)Ag + a + (long long)r * (np + 1)) +
                               (long long)jc * (np + 1))
                         : -CH_KV_MAX;
        }
        group_sync();  // sm.ld / sm.ls are read
    };
    // (staged: from shared memory)
    auto put_staged = [&](const Hot<EPL>& H, const ChOwn& own) CH_INLINE {
        const int q = warp % Cfg::LN;
#pragma unroll
        for (int e = 0; e < EPL; ++e) {
            const int x = (e * Cfg::LN + q) * 32 + lane;
            if (e * Cfg::LN * 32 > own.n) break;  // uniform
            sm.str[x] = H.r[e];
            sm.sta[x] = H.a[e] | ((H.pend >> e) & 1u ? (int)0x80000000 : 0);
            sm.stS[x] = H.Sb[e];
            sm.stk[x] = H.kv[e];
            sm.stK[x] = H.SK[e];
            sm.stb[x] = H.hb[e];
            sm.sty[x] = H.hy[e];
            sm.std_[x] = H.hd[e];
        }
        if (q == 0 && lane == 0) sm.sto = own;
    };
    auto get_staged = [&](Hot<EPL>& H, ChOwn& own) CH_INLINE {
        own = sm.sto;
        H.n = own.n;
        H.M = own.M;
        H.s = own.s;
        H.inv_s = own.inv_s;
        H.sumP = own.sumP;
        H.pend = 0;
#pragma unroll
        for (int e = 0; e < EPL; ++e) {
            const int x = elem(e);
            H.num[e] = H.sg[e] = f_inf();
            H.r[e] = H.a[e] = H.Sb[e] = 0;
            H.SK[e] = 0;
            H.kv[e] = -CH_KV_MAX;
            set_consts(H, e, f_inf(), 0.0f, 0.0f, 0);
            if (x >= own.n) continue;
            const int a = sm.sta[x];
            H.r[e] = sm.str[x];
            H.a[e] = a & 0x7fffffff;
            H.pend |= (unsigned)(a < 0) << e;
            H.Sb[e] = sm.stS[x];
            H.kv[e] = sm.stk[x];
            H.SK[e] = sm.stK[x];
            set_consts(H, e, sm.stb[x], sm.sty[x], sm.std_[x], sat((long long)hc * H.r[e]));
        }
    };

    // whether this warp's requests admit the candidate
    auto test = [&](const Hot<EPL>& H, const CandRec& cq, int a_in, auto ea) CH_INLINE {
        constexpr int EA = decltype(ea)::value;
        const float a = cq.a;
        const int ri = cq.ri;
        // KV usage allowed at a request's last iteration: M, less the
        // candidate's own share if it is still running then
        const long long Mll = (long long)H.M - jc - (long long)hc * a_in;
        const int Ma = Mll < -1 ? -1 : (int)Mll;
        bool ok = true;
        float mS = f_inf(), mSp = f_inf(), mv = f_inf();
#pragma unroll
        for (int e = 0; e < EA; ++e) {
            const bool le = H.r[e] <= ri, pe = (H.pend >> e) & 1u;
            ok = ok & ((le ? H.hh[e] : 0) + H.kv[e] <= (le ? Ma : H.M));
            // the quotient num / cost >= a: where num - a cost >= 0 it holds
            const float v = fmaf(-a, H.hd[e], H.num[e]);
            mv = fminf(mv, le ? v : f_inf());
            mS = fminf(mS, le | pe ? f_inf() : H.sg[e]);
            mSp = fminf(mSp, le | !pe ? f_inf() : H.sg[e]);
        }
        if (P.approx) return __all_sync(FULL, ok) != 0;
        const float f1 = fmaf(row_gt(mS, H.inv_s, H.stallk), cq.inv_d1, cq.nXd1);
        const float f2 = fmaf(mSp * H.inv_s, cq.inv_d2, cq.Ua);
        ok = ok & (f1 - a >= 0.0f) & (f2 >= 0.0f);
        if (__all_sync(FULL, ok & (mv >= 0.0f))) return true;
        // short somewhere: only of quotients that may still round up to a?
        bool maybe = ok;
#pragma unroll
        for (int e = 0; e < EA; ++e) {
            const float d = H.hd[e];
            maybe = maybe & (H.r[e] > ri || H.r[e] == 0 ||
                             fmaf(-a, d, H.num[e]) >= -(a * d * 2.4e-7f + 1e-30f));
        }
        if (!__all_sync(FULL, maybe)) return false;
#pragma unroll
        for (int e = 0; e < EA; ++e)
            if (H.r[e] > 0 && H.r[e] <= ri) ok = ok & (H.num[e] / H.hd[e] >= a);
        return __all_sync(FULL, ok) != 0;
    };
    // bounds of a request of aggregates Sb, SK (finishing before / after the
    // candidate), for pending prompts sumP
    auto bounds = [&](const Hot<EPL>& H, int r, int Sb, long long SK, float hb, float hy, bool pe,
                      float stallk, float& num, float& sg) CH_INLINE {
        const float T = decode_time(P, H.s, (float)r, (float)Sb, (float)SK);
        const float sigma = hb - T;
        const float u = shared_slack(H.s, sigma, hy);
        sg = sigma;
        num = pe ? u : stalled_slack(H.s, u, stallk);
    };
    // the aggregates with a request of prompt a and output r added
    auto add_to = [&](int re, int a, int r, int& Sb, long long& SK) CH_INLINE {
        const int m = min(re, r);
        Sb += m;
        SK += (long long)((unsigned)m * (unsigned)a + tri32(m));
    };

    // One link of a hot warp, candidate k (cq, rw): vote on it and, while the
    // decision is made, form candidate k + 2's partial sums and this slot's
    // state with candidate k appended; take it over if the decision is this
    // slot. won: the slot took candidate k - 1. Returns the decision; cq and rw
    // become candidate k + 1's.
    auto link = [&](Hot<EPL>& H, int k, bool won, CandRec& cq, int4& rw, auto ea) CH_INLINE {
        constexpr int EA = decltype(ea)::value;
        const int b = k & (CH_RING - 1), par = k & 1;
        const bool ok = H.n > 0 && test(H, cq, rw.x, ea);
        if (lane == 0) sm.vote[par][warp] = ok ? 1u : 0u;
        votes_sync();
        const ChElem ne = sm.ne[par][hs][won ? 1 : 0];
        const float4 rcv = sm.rc[b];
        const CandRec cq1 = sm.rec[(k + 1) & (CH_RING - 1)];
        const int4 rw1 = sm.raw[(k + 1) & (CH_RING - 1)];
        const int ri2 = sm.rec[(k + 2) & (CH_RING - 1)].ri;
        const int a = rw.x, r = rw.y, n0 = H.n;
        const int ha = sat((long long)hc * a) + jc;
        const float stallk = stall_terms(P, (float)(H.sumP + a));
        const float cost = prompt_cost_new(P, H.s, cq.r);
        const int hr = sat((long long)hc * r);
        int Sb[EA], kv[EA];
        long long SK[EA];
        float num[EA], sg[EA];
#pragma unroll
        for (int e = 0; e < EA; ++e) {
            const bool fresh = elem(e) == n0;
            Sb[e] = H.Sb[e];
            SK[e] = H.SK[e];
            add_to(H.r[e], a, r, Sb[e], SK[e]);
            // (unsigned)(r[e] - 1) < r: 1 <= r[e] <= r
            kv[e] = (unsigned)(H.r[e] - 1) < (unsigned)r
                        ? min(CH_KV_MAX, H.kv[e] + ha + H.hh[e])
                        : H.kv[e];
            Sb[e] = fresh ? ne.Sb : Sb[e];
            SK[e] = fresh ? ne.SK : SK[e];
            kv[e] = fresh ? ne.kv : kv[e];
            bounds(H, fresh ? r : H.r[e], Sb[e], SK[e], fresh ? rcv.y : H.hb[e],
                   fresh ? rcv.z : H.hy[e], fresh || ((H.pend >> e) & 1u), stallk, num[e],
                   sg[e]);
        }
        partial_sums(H, ri2, par, ea);
        decision_wait();
        const int d = sm.dec[par];
        if (d == hs) {
#pragma unroll
            for (int e = 0; e < EA; ++e) {
                H.Sb[e] = Sb[e];
                H.SK[e] = SK[e];
                H.kv[e] = kv[e];
                H.num[e] = num[e];
                H.sg[e] = sg[e];
                const bool fresh = elem(e) == n0;
                H.r[e] = fresh ? r : H.r[e];
                H.a[e] = fresh ? a : H.a[e];
                H.pend |= fresh ? 1u << e : 0u;
                H.hb[e] = fresh ? rcv.y : H.hb[e];
                H.hy[e] = fresh ? rcv.z : H.hy[e];
                H.hd[e] = fresh ? cost : H.hd[e];
                H.hh[e] = fresh ? hr : H.hh[e];
            }
            H.n = n0 + 1;
            H.sumP += a;
            H.stallk = stallk;
        }
        cq = cq1;
        rw = rw1;
        return d;
    };

    // CH_TERMS: lane (slot, version) forms whether worker `o`'s own terms admit
    // candidate k and what the candidate's aggregates on it would be, for the
    // worker as it is (version 0) and with candidate k - 1 appended (1). late:
    // the slot took candidate k - 2 after its partial sums were formed.
    auto terms = [&](const ChOwn& o, int k, bool with_prev, bool late) CH_INLINE {
        const int par = k & 1, slot = lane >> 1, ver = lane & 1;
        if (slot >= KH) return;
        const CandRec cq = sm.rec[k & (CH_RING - 1)];
        const int4 rw = sm.raw[k & (CH_RING - 1)];
        ChSums t = slot_sums(slot, par);
        auto add = [&](const int4 pw, bool on) {
            const bool gt = pw.y > cq.ri;
            t.n += on & gt ? 1 : 0;
            t.A += on & gt ? pw.x : 0;
            t.PR += on & !gt ? pw.y : 0;
            t.PRA += on & !gt ? (unsigned)pw.y * (unsigned)pw.x + tri32(pw.y) : 0u;
        };
        add(sm.raw[(k - 2) & (CH_RING - 1)], late);
        ChOwn w = o;
        const bool on = ver && with_prev;
        const int4 pw = sm.raw[(k - 1) & (CH_RING - 1)];
        add(pw, on);
        w.n += on ? 1 : 0;
        w.sumP += on ? pw.x : 0;
        w.npend += on ? 1 : 0;
        w.sumIn += on ? pw.x : 0;
        w.sumPred += on ? pw.y : 0;
        w.wpmax = on ? fmaxf(w.wpmax, sm.rc[(k - 1) & (CH_RING - 1)].x) : w.wpmax;
        const float a = cq.a;
        const int ri = cq.ri;
        bool ok = (long long)w.M - (long long)jc * (t.n + 1) >=
                  (long long)hc * ((long long)t.A + (long long)ri * (t.n + 1) + rw.x);
        const float4 wr = worker_record(P, w.inv_s, w.off, (float)w.sumP, w.wpmax, w.npend);
        ok = ok & (fminf(fmaf(cq.Zc, wr.x, -wr.y), wr.z) - a >= 0.0f);
        if (P.approx) {
            if (w.w != NONE) {
                const float2 wa = approx_bounds(P, C.scaled[w.w], w.dmin, w.n, w.sumP, w.sumIn,
                                                w.sumPred);
                ok = ok & (wa.x - a >= 0.0f) & (wa.y - cq.Ua >= 0.0f);
            }
        } else {
            const float nf = (float)t.n;
            const float b1 = row_b1(P, w.inv_s, nf, (float)t.A);
            const float b0n = row_b0n(P, (float)t.PR, (float)t.PRA);
            ok = ok & (fmaf(b0n, cq.inv_r, fmaf(-0.5f * nf, cq.r, cq.Ua - b1)) >= 0.0f);
        }
        sm.own_ok[par][slot][ver] = ok ? 1u : 0u;
        sm.ne[par][slot][ver] = new_elem(t, rw.x, rw.y);
    };

    // The last look-ahead warp: the outcomes of candidates [k0, k1), at most 32,
    // logged by the links, written a lane each.
    unsigned long long placed = 0, failed = 0;  // trace mode (the same in every lane)
    int keep = 0;                               // trace mode: waiting list
    auto flush = [&](int k0, int k1) CH_INLINE {
        const int k = k0 + lane, b = k & (CH_RING - 1);
        const bool on = k < k1;
        const int w = on ? sm.lw_[b] : 0;
        if (on && w >= 0) {  // the request in its worker's next slot
            const long long slot = (long long)w * cap + sm.ln[b];
            const int4 rw = sm.raw[b];
            C.in[slot] = rw.x;
            C.gen[slot] = 0;
            C.pred[slot] = rw.y;
            C.real[slot] = rw.z;
            C.tdec[slot] = 0.0;
            C.pend[slot] = 1;
            C.wait[slot] = sm.wd[b];
        }
        if (!sim) {
            if (on) io.placement[c0 + k * G] = w;
            return;
        }
        if (on && io.sim_pl) {
            io.sim_pl[k] = w;
            io.sim_tix[k] = sm.tix[b];
        }
        placed += __popc(__ballot_sync(FULL, on && w >= 0));
        bool fails = false;
        if (on && w < 0) {
            const double tau_alone = C.scaled[0] * (P.k1d * (double)sm.raw[b].x + P.c1d);
            // a decode instance has no TTFT budget to absorb a wait
            fails = w == -2 || P.decode || sm.wd[b] + io.H + tau_alone > P.T_pred;
        }
        failed += __popc(__ballot_sync(FULL, fails));
        const unsigned waits = __ballot_sync(FULL, on && w < 0 && !fails);
        if ((waits >> lane) & 1u) io.wl[keep + __popc(waits & ((1u << lane) - 1u))] = sm.tix[b];
        keep += __popc(waits);
    };

    // The worker of this slot leaves: its table from its requests' aggregates
    // (the same values that a table build forms by sorting and summing), its
    // sorted keys, record and key, and its entries among the modified workers.
    // The requests it held when it was loaded are in sorted order already; the
    // later ones are inserted.
    auto leave_with = [&](const Hot<EPL>& H, auto en) CH_INLINE {
        constexpr int EA = decltype(en)::value;  // elements a lane that may be in use
        const ChOwn own = sm.own[hs];
        const int w = own.w, m = own.m, n = H.n, n0 = sm.hn[hs], ins = n - n0;
        const long long base = (long long)w * cap, rowbase = (long long)w * C.rows;
        const float rank_bits = C.wrec[w].w;
        const int pad = (ins + 3) & ~3;
        unsigned key[EA];
        int at[EA];
#pragma unroll
        for (int e = 0; e < EA; ++e) {
            const int x = elem(e);
            key[e] = x < n0 ? C.skey[base + x]
                            : x < n ? ((unsigned)H.r[e] << 10) | (unsigned)x : 0xffffffffu;
            if (x < n0) sm.okey[x] = key[e];
            else if (x < n0 + pad) sm.nkey[x - n0] = key[e];
        }
        for (int j = ins + q * 32 + lane; j < pad; j += 32 * NWG) sm.nkey[j] = 0xffffffffu;
        hot_group_sync<NWG>();
#pragma unroll
        for (int e = 0; e < EA; ++e) {
            const int x = elem(e);
            at[e] = x;
            if (x >= n0 && x < n) {
                int lo = 0, hi = n0;
                while (lo < hi) {
                    const int mid = (lo + hi) >> 1;
                    if (sm.okey[mid] < key[e]) lo = mid + 1;
                    else hi = mid;
                }
                at[e] = lo;
            }
        }
        for (int k = 0; k < pad / 4; ++k) {
            const uint4 v = reinterpret_cast<const uint4*>(sm.nkey)[k];
#pragma unroll
            for (int e = 0; e < EA; ++e)
                at[e] += (v.x < key[e]) + (v.y < key[e]) + (v.z < key[e]) + (v.w < key[e]);
        }
#pragma unroll
        for (int e = 0; e < EA; ++e)
            if (elem(e) < n) {
                const int p = at[e];
                sm.key[p] = key[e];
                sm.ea[p] = H.a[e] | ((H.pend >> e) & 1u ? (int)0x80000000 : 0);
                sm.ekv[p] = H.kv[e];
                sm.eSb[p] = H.Sb[e];
                sm.eSK[p] = H.SK[e];
                sm.ebnd[p] = H.num[e] / H.hd[e];
                sm.esg[p] = H.sg[e];
            }
        hot_group_sync<NWG>();
        // sorted element elem(e) from here on: scans inside the chunk of 32
        // (prefix: rows, KV peak with h r, bounds of ongoing and new requests;
        // suffix, exclusive: KV peak, context, slacks), then over the chunks
        int r[EA], rows[EA], pk[EA], sk[EA], sa[EA];
        float po[EA], pn[EA], so[EA], sn[EA];
        unsigned last = 0;
#pragma unroll
        for (int e = 0; e < EA; ++e) {
            const int x = elem(e);
            const bool on = x < n;
            const unsigned k = on ? sm.key[x] : 0u;
            r[e] = (int)(k >> 10);
            const int a = on ? sm.ea[x] : 0;
            const float bnd = on ? sm.ebnd[x] : f_inf(), sg = on ? sm.esg[x] : f_inf();
            rows[e] = on && (x == 0 || (int)(sm.key[x - 1] >> 10) != r[e]) ? 1 : 0;
            if (on && (x == n - 1 || (int)(sm.key[x + 1] >> 10) != r[e])) last |= 1u << e;
            sk[e] = on ? sm.ekv[x] : -CH_KV_MAX;
            // (every hot worker's KV usage stays within M < 2^24)
            pk[e] = on ? (int)min((long long)CH_KV_MAX, (long long)hc * r[e] + sk[e]) : -CH_KV_MAX;
            sa[e] = a & 0x7fffffff;
            po[e] = a < 0 ? f_inf() : bnd;
            pn[e] = a < 0 ? bnd : f_inf();
            so[e] = a < 0 ? f_inf() : sg;
            sn[e] = a < 0 ? sg : f_inf();
            if (on) C.skey[base + x] = k;
        }
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const bool up = lane >= d, dn = lane + d < 32;
#pragma unroll
            for (int e = 0; e < EA; ++e) {
                const int u0 = __shfl_up_sync(FULL, rows[e], d), u1 = __shfl_up_sync(FULL, pk[e], d);
                const float u2 = __shfl_up_sync(FULL, po[e], d), u3 = __shfl_up_sync(FULL, pn[e], d);
                const int d0 = __shfl_down_sync(FULL, sk[e], d), d1 = __shfl_down_sync(FULL, sa[e], d);
                const float d2 = __shfl_down_sync(FULL, so[e], d), d3 = __shfl_down_sync(FULL, sn[e], d);
                rows[e] += up ? u0 : 0;
                pk[e] = up ? max(pk[e], u1) : pk[e];
                po[e] = up ? fminf(po[e], u2) : po[e];
                pn[e] = up ? fminf(pn[e], u3) : pn[e];
                sk[e] = dn ? max(sk[e], d0) : sk[e];
                sa[e] += dn ? d1 : 0;
                so[e] = dn ? fminf(so[e], d2) : so[e];
                sn[e] = dn ? fminf(sn[e], d3) : sn[e];
            }
        }
#pragma unroll
        for (int e = 0; e < EA; ++e) {
            const int ch = e * NWG + q;
            if (lane == 31) {
                sm.ti[0][ch] = rows[e];
                sm.ti[1][ch] = pk[e];
                sm.tf[0][ch] = po[e];
                sm.tf[1][ch] = pn[e];
            }
            if (lane == 0) {
                sm.ti[2][ch] = sk[e];
                sm.ti[3][ch] = sa[e];
                sm.tf[2][ch] = so[e];
                sm.tf[3][ch] = sn[e];
            }
        }
        hot_group_sync<NWG>();
        const bool cl = lane < EA * NWG;
        int c_rows = cl ? sm.ti[0][lane] : 0, c_pk = cl ? sm.ti[1][lane] : -CH_KV_MAX;
        int c_sk = cl ? sm.ti[2][lane] : -CH_KV_MAX, c_sa = cl ? sm.ti[3][lane] : 0;
        float c_po = cl ? sm.tf[0][lane] : f_inf(), c_pn = cl ? sm.tf[1][lane] : f_inf();
        float c_so = cl ? sm.tf[2][lane] : f_inf(), c_sn = cl ? sm.tf[3][lane] : f_inf();
#pragma unroll
        for (int d = 1; d < EA * NWG; d <<= 1) {
            const bool up = lane >= d, dn = lane + d < 32;
            const int u0 = __shfl_up_sync(FULL, c_rows, d), u1 = __shfl_up_sync(FULL, c_pk, d);
            const float u2 = __shfl_up_sync(FULL, c_po, d), u3 = __shfl_up_sync(FULL, c_pn, d);
            const int d0 = __shfl_down_sync(FULL, c_sk, d), d1 = __shfl_down_sync(FULL, c_sa, d);
            const float d2 = __shfl_down_sync(FULL, c_so, d), d3 = __shfl_down_sync(FULL, c_sn, d);
            c_rows += up ? u0 : 0;
            c_pk = up ? max(c_pk, u1) : c_pk;
            c_po = up ? fminf(c_po, u2) : c_po;
            c_pn = up ? fminf(c_pn, u3) : c_pn;
            c_sk = dn ? max(c_sk, d0) : c_sk;
            c_sa += dn ? d1 : 0;
            c_so = dn ? fminf(c_so, d2) : c_so;
            c_sn = dn ? fminf(c_sn, d3) : c_sn;
        }
        const int R = __shfl_sync(FULL, c_rows, EA * NWG - 1);
        const int tot_a = __shfl_sync(FULL, c_sa, 0), SM0 = __shfl_sync(FULL, c_sk, 0);
        const float smS0 = __shfl_sync(FULL, c_so, 0), smSp0 = __shfl_sync(FULL, c_sn, 0);
        const long long sumP = own.sumP;
        // a table row of lengths [rho, next): stored, sampled, and the limits
        // of the lengths in it
        auto put_row = [&](int row, int rho_p, int next, const RowVals& o) CH_INLINE {
            store_row(C, rowbase + row, o, false);
            const int q1 = row + 1, i = (q1 >> shift) - 1;
            if (row < R && i >= 0 && i < rc && (q1 & ((1 << shift) - 1)) == 0)
                rho[(long long)m * rs + i] = (unsigned short)(next - 1);
            if (nub > 0) {
                float v = o.v0.y;
                if (!P.approx) v = fminf(v, fminf(o.v1.z, o.ext.x));
                int u = rho_p < 1 ? 0 : ub_index(rho_p);
                if (ub_least(u) < rho_p) ++u;
                for (; u < CH_UB && ub_least(u) < next; ++u) mub[m * nub + u] = v;
            }
        };
#pragma unroll
        for (int e = 0; e < EA; ++e) {
            const int ch = e * NWG + q, x = elem(e);
            const int before = ch > 0 ? ch - 1 : 0, after = ch + 1 < EA * NWG ? ch + 1 : ch;
            const bool hasb = ch > 0, hasa = ch + 1 < EA * NWG;
            const int o0 = __shfl_sync(FULL, c_rows, before), o1 = __shfl_sync(FULL, c_pk, before);
            const float o2 = __shfl_sync(FULL, c_po, before), o3 = __shfl_sync(FULL, c_pn, before);
            const int a0 = __shfl_sync(FULL, c_sk, after), a1 = __shfl_sync(FULL, c_sa, after);
            const float a2 = __shfl_sync(FULL, c_so, after), a3 = __shfl_sync(FULL, c_sn, after);
            // exclusive in the chunk
            const int e0 = __shfl_down_sync(FULL, sk[e], 1), e1 = __shfl_down_sync(FULL, sa[e], 1);
            const float e2 = __shfl_down_sync(FULL, so[e], 1), e3 = __shfl_down_sync(FULL, sn[e], 1);
            const bool in = lane < 31;
            if (!((last >> e) & 1u)) continue;
            const int row = rows[e] + (hasb ? o0 : 0);
            const int PM = hasb ? max(pk[e], o1) : pk[e];
            const float pmA = hasb ? fminf(po[e], o2) : po[e], pmAp = hasb ? fminf(pn[e], o3) : pn[e];
            const int SMx = max(in ? e0 : -CH_KV_MAX, hasa ? a0 : -CH_KV_MAX);
            const long long Ag = (in ? e1 : 0) + (hasa ? a1 : 0);
            const float smS = fminf(in ? e2 : f_inf(), hasa ? a2 : f_inf());
            const float smSp = fminf(in ? e3 : f_inf(), hasa ? a3 : f_inf());
            const int np = n - (x + 1), rr = r[e];
            const long long PR = sm.eSb[x] - (long long)rr * np;
            const long long PRA = sm.eSK[x] - (long long)np * tri32(rr) - (long long)rr * Ag;
            const int next = x == n - 1 ? 0x7fffffff : (int)(sm.key[x + 1] >> 10);
            const RowVals o = make_row(P, H.inv_s, H.M, sumP, rr, next, np, Ag, PR, PRA, PM,
                                       SMx == -CH_KV_MAX ? 0 : SMx, pmA, pmAp, smS, smSp);
            put_row(row, rr, next, o);
        }
        // row 0, the worker's record, and its key: a warp each
        if (q == NWG - 1 && lane == 31) {
            const int r0 = (int)(sm.key[0] >> 10);
            const RowVals o = make_row(P, H.inv_s, H.M, sumP, 0, r0, n, tot_a, 0, 0, LL_NONE, SM0,
                                       f_inf(), f_inf(), smS0, smSp0);
            put_row(0, 0, r0, o);
            C.R[w] = R;
            mR[m] = R;
        } else if (q == 0 && lane == 0) {
            float4 wr = worker_record(P, H.inv_s, own.off, (float)own.sumP, own.wpmax, own.npend);
            wr.w = rank_bits;
            C.wrec[w] = wr;
            mwrec[m] = wr;
        } else if (q == 1 && lane == 0) {
            const unsigned long long kq = hot_key(n, own.sumIn, own.sumPred);
            C.key[w] = kq;
            mkey[m] = kq;
            if (P.approx)
                C.wapx[w] = approx_bounds(P, C.scaled[w], own.dmin, n, own.sumP, own.sumIn,
                                          own.sumPred);
            sm.left_n = n;
        }
        hot_group_sync<NWG>();  // the scratch is free
    };

    auto leave = [&](const Hot<EPL>& H) CH_INLINE {
        if constexpr (EPL >= 4) {
            if (H.n <= EPL / 4 * 32 * NWG) return leave_with(H, IntC<EPL / 4>());
            if (H.n <= EPL / 2 * 32 * NWG) return leave_with(H, IntC<EPL / 2>());
        }
        leave_with(H, IntC<EPL>());
    };

    // Every role runs the same sequence of phases, each in a loop of its own
    // (one role's registers are not live in another's code): look ahead if
    // nothing is, links beside more look-ahead, and after a miss the change of
    // places. cta_sync parts the phases, and what a role decides for itself in
    // one (who stages the new worker, say) it decides from words that no role
    // writes in it: counts come from sm.miss_n and mn, never from C.n, which is
    // only written here. Of the modified workers' entries mw, mn and modbits are
    // the look-ahead warps' own, written in a change only; the rest of a slot is
    // written by the hot warps whose worker leaves, while mn says that it is hot
    // and nobody looks at it. Inside the links' phase votes_sync and the decision's
    // barrier order the double-buffered words; sm.abort alone is polled.
    int alt_end = 0, span = CH_SCAN;
    const int first = sim ? CH_FIRST : CH_SCAN;
    int stop_at = n_cand;
    // at the end the hot workers' tables are brought up to date (a simulation's
    // next step rebuilds every table, unless Algorithm 2 reads them first)
    const bool last_tables = n_cand > 0 && (!sim || io.sim_pl);
    if (warp < CH_HOT) {
        Hot<EPL> H;
        H.n = 0;
        H.M = H.sumP = 0;
        H.s = H.inv_s = 1.0f;
        H.stallk = 0.0f;
        H.pend = 0;
#pragma unroll
        for (int e = 0; e < EPL; ++e) {
            H.r[e] = H.a[e] = H.Sb[e] = 0;
            H.kv[e] = -CH_KV_MAX;
            H.SK[e] = 0;
            H.num[e] = H.sg[e] = f_inf();
            set_consts(H, e, f_inf(), 0.0f, 0.0f, 0);
        }
        bool won = false;
        CandRec cq;  // the next candidate
        int4 rw = make_int4(0, 0, 0, 0);
        for (int rp = 0; c < n_cand; rp ^= 1) {
            if (alt_end <= c) {
                cq = sm.rec[c & (CH_RING - 1)];
                rw = sm.raw[c & (CH_RING - 1)];
                with_elems(H.n, [&](auto ea) CH_INLINE {
                    partial_sums(H, cq.ri, c & 1, ea);
                    partial_sums(H, sm.rec[(c + 1) & (CH_RING - 1)].ri, (c + 1) & 1, ea);
                });
                won = false;
                alt_end = min(c + first, n_cand);
                span = sim ? CH_SCAN : CH_AHEAD;
                votes_sync();  // the sums are in: CH_TERMS forms candidate c's terms
                cta_sync();
            }
            int k = c, d = CH_NOBODY;
            while (k < alt_end && d != CH_END)
                with_elems(H.n + 1, [&](auto ea) CH_INLINE {
                    do {
                        d = link(H, k, won, cq, rw, ea);
                        won = d == hs;
                        ++k;
                    } while (k < alt_end && d != CH_END &&
                             H.n + 1 <= decltype(ea)::value * 32 * NWG);
                });
            if (d == CH_END && k < alt_end) votes_sync();  // CH_TERMS learns of it
            const int new_end = min(alt_end + span, n_cand);
            cta_sync();
            const int code = sm.code[rp];
            c = sm.next[rp];
            if (code == CH_DONE) {
                alt_end = new_end;
                span = CH_AHEAD;
                if (sm.slow[rp]) break;
                continue;
            }
            if (code == CH_STOP || sm.slow[rp]) break;
            // a miss at candidate c: worker w becomes hot in slot v
            const int w = sm.miss_w, f = sm.miss_f, v = sm.victim;
            if ((f & CH_UNMOD) && mcount == mmax) break;  // no room for another modified worker
            const int m = f & CH_UNMOD ? mcount++ : f & CH_IDX;
            if (hs == v) {
                const int b = c & (CH_RING - 1);
                rw = sm.raw[b];
                const float4 rcv = sm.rc[b];
                const int nw = sm.miss_n;
                const bool staged = Cfg::staged(nw, sim);
                if (sm.hw[v] != NONE) leave(H);
                ChOwn own;
                if (staged) {
                    staged_wait<Cfg::LN + NWG>();
                    get_staged(H, own);
                } else if constexpr (NWG > Cfg::LN) {
                    load(H, own, w, nw, IntC<NWG>());
                }
                const int n0 = H.n;
                with_elems(n0 + 1, [&](auto ea) CH_INLINE { partial_sums(H, rw.y, c & 1, ea); });
                hot_group_sync<NWG>();
                const ChElem ne = new_elem(slot_sums(hs, c & 1), rw.x, rw.y);
                const int ha = sat((long long)hc * rw.x) + jc;
                const float stallk = stall_terms(P, (float)(H.sumP + rw.x));
#pragma unroll
                for (int e = 0; e < EPL; ++e) {
                    const int x = elem(e);
                    if (e * NWG * 32 > n0) break;  // uniform
                    add_to(H.r[e], rw.x, rw.y, H.Sb[e], H.SK[e]);
                    if ((unsigned)(H.r[e] - 1) < (unsigned)rw.y)
                        H.kv[e] = min(CH_KV_MAX, H.kv[e] + ha + H.hh[e]);
                    if (x == n0) {
                        H.r[e] = rw.y;
                        H.a[e] = rw.x;
                        H.pend |= 1u << e;
                        H.Sb[e] = ne.Sb;
                        H.SK[e] = ne.SK;
                        H.kv[e] = ne.kv;
                        set_consts(H, e, rcv.y, rcv.z, prompt_cost_new(P, H.s, (float)rw.y),
                                   sat((long long)hc * rw.y));
                    }
                    bounds(H, H.r[e], H.Sb[e], H.SK[e], H.hb[e], H.hy[e],
                           (H.pend >> e) & 1u, stallk, H.num[e], H.sg[e]);
                }
                H.n = n0 + 1;
                H.sumP += rw.x;
                H.stallk = stallk;
                if (q == 0 && lane == 0) {
                    C.n[w] = n0 + 1;
                    sm.ln[b] = n0;
                    sm.hn[v] = n0;
                    own.m = m;
                    own.n += 1;
                    own.sumP += rw.x;
                    own.npend += 1;
                    own.sumIn += rw.x;
                    own.sumPred += rw.y;
                    own.wpmax = fmaxf(own.wpmax, rcv.x);
                    sm.own[v] = own;
                }
            }
            cta_sync();
            c += 1;
            alt_end = c;
        }
        cta_sync();  // (the other roles' last writes follow)
        if (last_tables) {
            cta_sync();  // the last links' logs and terms
            for (int k = 0; k < KH; ++k) {
                if (hs == k && sm.hw[k] != NONE) leave(H);
                cta_sync();
            }
        }
    } else if (warp == CH_DECIDE) {
        // lane i < KH: hot slot i's worker, its group, its key's terms, when it
        // last won, and how many of the hot workers come before it
        int hk_w = NONE, hk_m = 0, hk_g = 0, hk_n = 0, hk_in = 0, hk_pred = 0, hk_last = -1;
        int before = 0;
        unsigned long long hk_key = 0ull;
        auto rerank = [&]() {
            before = 0;
#pragma unroll
            for (int i = 0; i < KH; ++i) {
                const unsigned long long ok = __shfl_sync(FULL, hk_key, i);
                const int ow = __shfl_sync(FULL, hk_w, i);
                before += ok > hk_key || (ok == hk_key && ow < hk_w);
            }
        };
        int prev = CH_NOBODY;  // the slot that took the last candidate
        int took = 0;          // groups: candidates placed, and when the first was taken up
        const long long begun = A.placed_cost > 0 ? clock64() : 0;
        bool voted = false;    // this group's chain is the slower way
        for (int rp = 0; c < n_cand; rp ^= 1) {
            if (alt_end <= c) {
                rerank();
                prev = CH_NOBODY;
                alt_end = min(c + first, n_cand);
                span = sim ? CH_SCAN : CH_AHEAD;
                votes_sync();
                cta_sync();
            }
            int code = CH_DONE, k = c;
            for (; k < alt_end; ++k) {
                const int b = k & (CH_RING - 1), par = k & 1;
                const bool valid = sm.rec[b].valid != 0;
                const int4 rw = sm.raw[b];
                const unsigned long long ak = sm.alt_k[b];
                const int aw = sm.alt_w[b], af = sm.alt_f[b];
                // hot workers that come before the best of the others and may
                // take the candidate's group
                const bool may = lane < KH && hk_w != NONE && valid &&
                                 (aw == NONE || hk_key > ak || (hk_key == ak && hk_w < aw)) &&
                                 hk_g == rw.w;
                const unsigned full = __ballot_sync(FULL, hk_n >= cap);
                const unsigned rank = may ? (unsigned)before << 4 | (unsigned)lane : 0xffffffffu;
                const unsigned* own = &sm.own_ok[par][lane < KH ? lane : 0][prev == lane ? 1 : 0];
                const bool alt = valid && aw != NONE;
                votes_sync();
                const unsigned own_ok = *own;
                const unsigned votes =
                    __ballot_sync(FULL, lane < CH_HOT && sm.vote[par][lane & (CH_HOT - 1)] != 0);
                constexpr unsigned all = (1u << NWG) - 1u;
                // (a shift by lane % KH: the other lanes' rank keeps them out)
                const bool yes = own_ok != 0 && ((votes >> (lane % KH * NWG)) & all) == all;
                const unsigned pick = __reduce_min_sync(FULL, yes ? rank : 0xffffffffu);
                const bool hit = pick != 0xffffffffu;
                // a worker that is not hot, or that has no free slot, ends the run
                const bool end = hit ? ((full >> (pick & 15u)) & 1u) != 0 : alt;
                const int d = end ? CH_END : hit ? (int)(pick & 15u) : CH_NOBODY;
                if (lane == 0) sm.dec[par] = d;
                __syncwarp();
                decision_arrive();
                if (end) {
                    code = hit || (af & CH_FULL) ? CH_STOP : CH_MISS;
                    if (lane == 0) *(volatile int*)&sm.abort = 1;
                    if (k + 1 < alt_end) votes_sync();
                    break;
                }
                prev = d;
                if (!hit) {
                    if (lane == 0) sm.lw_[b] = valid ? -1 : -2;
                    continue;
                }
                ++took;
                const bool me = lane == d;
                if (me) sm.lw_[b] = hk_w;
                if (me) sm.ln[b] = hk_n;
                hk_n += me ? 1 : 0;
                hk_in += me ? rw.x : 0;
                hk_pred += me ? rw.y : 0;
                hk_last = me ? k : hk_last;
                hk_key = hk_w == NONE ? 0ull : hot_key(hk_n, hk_in, hk_pred);
                if (pick >> 4) {  // its key grew: it may come before others now
                    const unsigned long long kd = __shfl_sync(FULL, hk_key, d);
                    const int wd = __shfl_sync(FULL, hk_w, d), bd = (int)(pick >> 4);
                    const bool ahead = lane < KH && !me && (hk_key > kd || (hk_key == kd && hk_w < wd));
                    const unsigned who = __ballot_sync(FULL, ahead);
                    before = me ? __popc(who) : before + (!ahead && before < bd ? 1 : 0);
                }
            }
            const unsigned lru = __reduce_min_sync(
                FULL, lane < KH ? ((unsigned)(hk_last + 1) << 4) | (unsigned)lane : 0xffffffffu);
            const int b = k & (CH_RING - 1);
            if (lane < KH) {
                sm.hw[lane] = hk_w;
                sm.hm[lane] = hk_m;
                if (hk_w != NONE) C.n[hk_w] = hk_n;
            }
            if (lane == 0) {
                sm.code[rp] = code;
                sm.next[rp] = k;
                int slow = 0;
                if (A.placed_cost > 0 && k >= CH_TRIAL) {
                    if (!voted && clock64() - begun > (long long)took * A.placed_cost +
                                                          (long long)(k - took) * A.other_cost) {
                        voted = true;
                        atomicAdd(A.votes, 1);
                    }
                    slow = 2 * *(volatile int*)A.votes >= G;
                }
                sm.slow[rp] = slow;
                if (code == CH_MISS) {
                    const int w = sm.alt_w[b], f = sm.alt_f[b];
                    sm.miss_w = w;
                    sm.miss_f = f;
                    sm.victim = (int)(lru & 15u);
                    const int i = f & CH_IDX;
                    sm.miss_n = !(f & CH_UNMOD) ? mn[i] : i < nwin ? win[i].n : rank_ent[i].n;
                    sm.lw_[b] = w;
                } else if (code == CH_STOP) {
                    *io.status = -2;  // ALADDIN_ERR_CAPACITY
                    if (!sim)
                        for (int i = k; i < n_cand; ++i) io.placement[c0 + i * G] = -1;
                }
            }
            const int new_end = min(alt_end + span, n_cand);
            cta_sync();
            c = k;
            if (code == CH_DONE) {
                alt_end = new_end;
                span = CH_AHEAD;
                if (sm.slow[rp]) break;
                continue;
            }
            if (code == CH_STOP || sm.slow[rp]) break;
            const int f = sm.miss_f, v = sm.victim;
            if ((f & CH_UNMOD) && mcount == mmax) break;
            if (f & CH_UNMOD) mcount++;
            ++took;
            if (lane == 0) sm.abort = 0;
            cta_sync();
            if (lane == v) {
                const ChOwn& o = sm.own[v];
                hk_w = o.w;
                hk_m = o.m;
                hk_g = filter ? o.w % GP : 0;
                hk_n = o.n;
                hk_in = o.sumIn;
                hk_pred = o.sumPred;
                hk_key = hot_key(hk_n, hk_in, hk_pred);
                hk_last = c;
            }
            c += 1;
            alt_end = c;
        }
        cta_sync();  // the last phase's readers are done
        if (lane < KH) {
            sm.hw[lane] = hk_w;
            sm.hm[lane] = hk_m;
        }
    } else if (warp == CH_TERMS) {
        ChOwn o;  // lane (slot, version): the slot's worker
        o.w = NONE;
        o.m = o.n = o.M = o.sumP = o.npend = o.sumIn = o.sumPred = 0;
        o.s = o.inv_s = 1.0f;
        o.off = o.wpmax = 0.0f;
        o.dmin = 0.0;
        auto take = [&](int k) {  // candidate k went to the lane's slot
            const int4 pw = sm.raw[k & (CH_RING - 1)];
            o.n += 1;
            o.sumP += pw.x;
            o.npend += 1;
            o.sumIn += pw.x;
            o.sumPred += pw.y;
            o.wpmax = fmaxf(o.wpmax, sm.rc[k & (CH_RING - 1)].x);
        };
        bool owed = false;  // the slot took the last run's last candidate
        for (int rp = 0; c < n_cand; rp ^= 1) {
            if (alt_end <= c) {
                alt_end = min(c + first, n_cand);
                span = sim ? CH_SCAN : CH_AHEAD;
                votes_sync();
                terms(o, c, false, false);
                cta_sync();
                owed = false;
            }
            for (int k = c; k < alt_end; ++k) {
                votes_sync();
                bool late = owed;
                if (k > c) {
                    const int d = sm.dec[(k - 1) & 1];
                    if (d <= CH_END) break;
                    late = d == lane >> 1;
                    if (late) take(k - 1);
                }
                terms(o, k + 1, true, late);
                owed = false;
                __syncwarp();
            }
            const int new_end = min(alt_end + span, n_cand);
            if (!(lane & 1) && lane >> 1 < KH) sm.own[lane >> 1] = o;
            cta_sync();
            const int code = sm.code[rp];
            c = sm.next[rp];
            if (code == CH_DONE) {
                alt_end = new_end;
                span = CH_AHEAD;
                owed = sm.dec[(c - 1) & 1] == lane >> 1;
                if (owed) take(c - 1);
                if (sm.slow[rp]) break;
                continue;
            }
            if (code == CH_STOP || sm.slow[rp]) break;
            const int f = sm.miss_f, v = sm.victim;
            if ((f & CH_UNMOD) && mcount == mmax) break;
            if (f & CH_UNMOD) mcount++;
            cta_sync();
            if (lane >> 1 == v) o = sm.own[v];
            c += 1;
            alt_end = c;
        }
        cta_sync();  // the last phase's readers are done
        if (!(lane & 1) && lane >> 1 < KH) sm.own[lane >> 1] = o;
    } else {
        // a lane holds candidate k's look against the worker that left slot v
        auto hold_against = [&](int k, int v, int w) CH_INLINE {
            const int b = k & (CH_RING - 1);
            const int i = sm.hm[v], ow = sm.hw[v], n = sm.left_n;
            bool held = sm.alt_at[b] == k + 1;
            if (held && sm.alt_w[b] == w) {
                held = false;
                sm.alt_at[b] = 0;
            }
            const CandRec cq = sm.rec[b];
            if (held && ow != NONE && cq.valid && (!filter || ow % GP == sm.raw[b].w)) {
                const unsigned long long ok = mkey[i];
                if (sm.alt_w[b] == NONE || ok > sm.alt_k[b] ||
                    (ok == sm.alt_k[b] && ow < sm.alt_w[b])) {
                    const long long rb = (long long)ow * C.rows;
                    const long long row = rb + slot_row(i, rb, mR[i], cq.ri);
                    const float4* t = C.tab + row * ROW_F4;
                    float m;
                    if (eval_pair_mode(P.approx != 0, t[0], t[1], C.tab2[row], mwrec[i],
                                       P.approx ? C.wapx[ow] : make_float2(0.0f, 0.0f), cq,
                                       m) == 15u) {
                        sm.alt_k[b] = ok;
                        sm.alt_w[b] = ow;
                        sm.alt_f[b] = i | (n >= cap ? CH_FULL : 0);
                    }
                }
            }
            if (lane == 0 && ow != NONE) mn[i] = n;  // not hot any more
        };
        const bool clerk = warp == CH_WARPS - 1;  // fetches the records, writes the outcomes
        int written = 0;  // candidates whose outcomes are written
        bool change = false;  // in a change of the hot worker: slot v takes worker w
        int v = 0, w = NONE;
        for (int rp = 0; c < n_cand || change; rp ^= 1) {
            if (alt_end <= c) {
                // The next candidates. Looks made before stay right unless they found
                // the worker that is hot now (they are made again), but for the
                // worker that leaves, whose new table they are held against once it
                // is there. (Made afresh at every miss they cost rounds that use
                // many workers of large fleets up to half of their time: 218
                // candidates on 14,000 workers of 128 slots 2.0 ms, 1.44 so.)
                const int k = c + warp - (CH_WARPS - first);
                if (k >= c && k < n_cand &&
                    !(sm.alt_at[k & (CH_RING - 1)] == k + 1 && sm.alt_w[k & (CH_RING - 1)] != w))
                    look(k, &sm.never);
                if (change) {
                    cta_sync();
                    if (warp == CH_LOOK0) hold_against(c + lane, v, w);
                    change = false;
                    if (c >= n_cand) break;
                }
                alt_end = min(c + first, n_cand);
                span = sim ? CH_SCAN : CH_AHEAD;
                cta_sync();
            }
            const int new_end = min(alt_end + span, n_cand);
            const int rec_new = max(rec_end, min(n_cand, new_end + CH_AHEAD));
            if (clerk) {
                flush(written, c);  // (their records are in the ring until fetch takes their place)
                written = c;
                __syncwarp();
                for (int k = rec_end + lane; k < rec_new; k += 32) fetch(k);
            }
            if (A.F)
                for (int k = rec_end + warp - CH_LOOK0; k < rec_new; k += CH_SCAN) fetch_row(k);
            rec_end = rec_new;
            for (int k = alt_end + warp - CH_LOOK0; k < new_end; k += CH_SCAN) {
                if (sm.alt_at[k & (CH_RING - 1)] == k + 1) continue;
                if (__any_sync(FULL, *(volatile int*)&sm.abort)) break;
                look(k, &sm.abort);
            }
            cta_sync();
            const int code = sm.code[rp];
            c = sm.next[rp];
            if (code != CH_STOP && sm.slow[rp]) {
                stop_at = c;
                break;
            }
            if (code == CH_DONE) {
                alt_end = new_end;
                span = CH_AHEAD;
                continue;
            }
            if (code == CH_STOP) break;
            const int f = sm.miss_f;
            v = sm.victim;
            w = sm.miss_w;
            if ((f & CH_UNMOD) && mcount == mmax) {
                stop_at = c;
                break;
            }
            // hot from here on (bit 31), so that the look-ahead leaves it out
            if (warp == CH_LOOK0 && lane == 0) {
                mn[f & CH_UNMOD ? mcount : f & CH_IDX] = (int)0x80000000;
                if (f & CH_UNMOD) {
                    const int pos = f & CH_IDX;
                    mw[mcount] = w;
                    modbits[pos >> 5] |= 1u << (pos & 31);
                }
            }
            look_sync();
            if (f & CH_UNMOD) mcount++;
            // while the hot warps write the leaving worker's table: worker w is
            // staged (or its requests fetched into L1), and the next candidates
            // are looked at among the workers other than the leaving one
            const int nw = sm.miss_n;
            if (Cfg::staged(nw, sim)) {
                if (warp < CH_LOOK0 + Cfg::LN) {
                    Hot<EPL> H;
                    ChOwn own;
                    load(H, own, w, nw, IntC<Cfg::LN>());
                    put_staged(H, own);
                    staged_arrive<Cfg::LN + NWG>();
                }
            } else {
                const long long base = (long long)w * cap;
                for (int x = 32 * ((warp - CH_LOOK0) * 32 + lane); x < nw; x += 32 * 32 * CH_SCAN) {
                    const void* const line[] = {C.skey + base + x, C.in + base + x,
                                                C.gen + base + x, C.pred + base + x,
                                                C.bank + base + x, C.pend + base + x};
#pragma unroll
                    for (int i = 0; i < 6; ++i)
                        asm volatile("prefetch.global.L1 [%0];" ::"l"(line[i]));
                }
            }
            change = true;
            c += 1;
            alt_end = c;
        }
        cta_sync();  // (likewise)
        if (clerk) flush(written, c);
    }
    if (last_tables && warp >= CH_HOT)
        for (int k = 0; k <= KH; ++k) cta_sync();
    if (warp == CH_WARPS - 1 && lane == 0) {
        if (!sim) {
            if (A.c_stop) A.c_stop[g] = stop_at;
        } else {
            io.counters[0] += failed;
            io.counters[1] += placed;
            if (*io.status == 0) {
                if (io.sim_n) *io.sim_n = n_cand;
                *io.n_wait = keep;
                if (io.stop_at_fail && io.counters[0] > 0) {
                    *io.status = 1;
                    io.counters[2] = (unsigned long long)io.hb;
                }
            }
        }
    }
}

// Shared memory of k_round_chain: the fixed part, nwin rank entries, mmax
// modified workers of rc samples and nub limits, and the bit set of W rank
// positions.
template <int E>
static size_t ch_smem(int W, int nwin, int mmax, int rc, int nub, int nts = 0)
{
    const int nwords = (W + 31) >> 5;
    return ((sizeof(ChSmem<E>) + 15) / 16) * 16 + (size_t)nwin * sizeof(RankEnt) +
           (size_t)((nwords + 3) & ~3) * 4 +
           (size_t)mmax * (16 + 8 + 4 * 3 + 4 * (size_t)nub + 2 * (size_t)(rc + R2_RHO_PAD)) +
           (nts > 0 ? (size_t)W * 2 * (size_t)(nts + R2_RHO_PAD) : 0);
}

// Groups. A chain's looks evaluate 32 workers at a time where k_round_grp evaluates
// 512: on groups of a few hundred workers up the load decides which is faster
// (300 candidates a group: a half-empty fleet, whose looks end early, 600 workers
// of 128 slots a group, 3.5 ms with k_round_grp and 0.97 as a chain; nearly full
// ones, 700 a group 3.6 and 4.5, 3,000 of 1,024 slots 22.9 and 51). So past the line
// up to which the chain leads every group times itself against what k_round_grp
// takes for the same candidates, and when half of the groups have taken half as
// long again all leave the rest to it (both place alike and leave the same tables;
// one group alone would wait for the others' chains first). The cycles: an
// evaluation of every 512 workers 3,900 and a fixed 4,000, and a table's rebuild
// (measured on 256 to 700 workers).
static void ch_group_costs(int cap, int W, int* placed, int* other)
{
    const int line = cap <= 32 ? 160 : cap <= 64 ? 224 : cap == 512 ? 416 : 320;
    if (W <= line) return;
    *other = 4000 + 3900 * ((W + 511) / 512);
    *placed = *other + (cap <= 32 ? 5500 : cap <= 64 ? 7000 : 10500);
    *other += *other / 2;
    *placed += *placed / 2;
}

struct ChPlan {
    int nwin, mmax, rc, nub, nts;
};

// W workers a chain; all: every one of them may be modified (no hand-off).
template <int E>
static bool ch_plan(int W, int cap, int K, int smem_max, bool sim, bool all, bool flags, ChPlan* p)
{
    if (K > 65536) return false;  // breakpoint samples are 16-bit
    const size_t budget = (size_t)smem_max - 1024;
    p->nwin = W < CH_WIN ? W : CH_WIN;
    if (sim) {  // ranked in shared memory: a power of two
        if (W > CH_SORT_MAX) return false;
        p->nwin = 1;
        while (p->nwin < W) p->nwin <<= 1;
    }
    const int rc_max = cap < CH_RC_MAX ? cap : CH_RC_MAX;
    const int most = W < CH_MAX_SLOTS ? W : CH_MAX_SLOTS;
    if (all && most < W) return false;
    // fewer samples, then no limits, before fewer workers
    for (int nub = CH_UB + 1; nub >= 0; nub -= CH_UB + 1)
        for (int rc = rc_max; rc >= 0; rc -= 16)
            if (ch_smem<E>(W, p->nwin, most, rc, nub) <= budget) {
                p->mmax = most;
                p->rc = rc;
                p->nub = nub;
                // (a fleet that a round modifies in full is rare)
                if (!all && rc < rc_max) continue;
                // without flags: samples of every worker with what is left
                p->nts = flags ? 0 : (cap >> CH_TSHIFT) < CH_TS_MAX ? cap >> CH_TSHIFT : CH_TS_MAX;
                while (p->nts > 0 && ch_smem<E>(W, p->nwin, most, rc, nub, p->nts) > budget)
                    p->nts -= 2;
                return true;
            }
    if (all) return false;
    const size_t base = ch_smem<E>(W, p->nwin, 0, 0, 0);
    const size_t per = ch_smem<E>(W, p->nwin, 1, rc_max, CH_UB + 1) - base;
    if (budget < base + 16 * per) return false;
    p->nts = 0;
    p->mmax = (int)std::min<size_t>((budget - base) / per, (size_t)most);
    p->rc = rc_max;
    p->nub = CH_UB + 1;
    return true;
}

template <int E>
cudaError_t round_chain_e(const DevParams& P, const ClusterDev& C, const RoundIO& io,
                                 const RoundChainBuffers* B, cudaStream_t st, bool* used)
{
    *used = false;
    DevInfo d;
    cudaError_t e = device_info(&d);
    if (e != cudaSuccess) return e;
    const int G = !io.sim && P.groups > 1 ? P.groups : 1;
    const int Wl = (C.W + G - 1) / G;
    const bool all = io.sim || G > 1;
    ChPlan pl;
    if (!ch_plan<E>(Wl, C.cap, P.K, d.smem_optin, io.sim != 0, all, !all && B->flags, &pl))
        return cudaSuccess;
    if (!all && P.round_slots_max > 0 && pl.mmax > P.round_slots_max) pl.mmax = P.round_slots_max;
    const size_t smem = ch_smem<E>(Wl, pl.nwin, pl.mmax, pl.rc, pl.nub, pl.nts);
    ChArgs A;
    A.P = P;
    A.C = C;
    A.io = io;
    A.F = nullptr;
    A.ldf = 0;
    A.rank_ent = B ? reinterpret_cast<RankEnt*>(B->rank) : nullptr;
    A.c_stop = io.sim ? nullptr : B->c_stop;
    A.placed_cost = A.other_cost = 0;
    A.mmax = pl.mmax;
    A.rc = pl.rc;
    A.nub = pl.nub;
    A.nwin = pl.nwin;
    A.nts = pl.nts;
    if ((e = allow_max_smem<k_round_chain<E>>()) != cudaSuccess) return e;
    *used = true;
    if (all) {
        if (G > 1) ch_group_costs(C.cap, Wl, &A.placed_cost, &A.other_cost);
        A.votes = A.placed_cost > 0 ? B->c_stop + G : nullptr;
        if (A.votes && (e = cudaMemsetAsync(A.votes, 0, sizeof(int), st)) != cudaSuccess) return e;
        k_round_chain<E><<<G, CH_THREADS, smem, st>>>(A);
        if ((e = cudaGetLastError()) != cudaSuccess || A.placed_cost == 0) return e;
        RoundIO rest = io;  // (nothing where every candidate was placed)
        rest.c_first = B->c_stop;
        return launch_round_groups(P, C, rest, st);
    }
    const int ldf = round_flag_row(C.W);
    int chunk = io.n_cand;
    if (B->flags) chunk = std::min(chunk, B->chunk);
    if (P.round_chunk > 0 && chunk > P.round_chunk) chunk = P.round_chunk;
    const bool fresh = B->flags && P.round_slots_max <= 0 && pl.mmax > CH_FRESH && chunk > CH_FRESH;
    if (fresh) A.mmax = pl.mmax = CH_FRESH;
    for (int c0 = 0, placed = 0; c0 < io.n_cand; c0 += placed) {
        const int n = std::min(chunk, io.n_cand - c0);
        placed = n;
        if (c0 > 0 && (e = launch_rank(C, st)) != cudaSuccess) return e;  // the chunk's start state
        A.io.in = io.in + c0;
        A.io.pred = io.pred + c0;
        A.io.wait = io.wait ? io.wait + c0 : nullptr;
        A.io.placement = io.placement + c0;
        A.io.n_cand = n;
        if (B->flags) {
            // every candidate of the chunk against the current state, rank order
            e = launch_score(P, C, n, A.io.in, A.io.pred, A.io.wait, B->flags, nullptr, nullptr,
                             nullptr, nullptr, B->score, io.round_open || c0 > 0, st, nullptr,
                             nullptr, false, C.order, ldf);
            if (e != cudaSuccess) return e;
            A.F = B->flags;
            A.ldf = ldf;
        }
        k_round_chain<E><<<1, CH_THREADS, smem, st>>>(A);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        if (fresh) {
            e = cudaMemcpyAsync(&placed, B->c_stop, sizeof(int), cudaMemcpyDeviceToHost, st);
            if (e != cudaSuccess || (e = cudaStreamSynchronize(st)) != cudaSuccess) return e;
            if (placed <= 0) return cudaErrorUnknown;  // (a chain places CH_FRESH at least)
        } else if (pl.mmax < C.W) {
            // the sliced round places what the chain left (nothing when every
            // candidate was placed: it returns at once)
            RoundIO rest = A.io;
            rest.c_first = B->c_stop;
            if ((e = launch_round(P, C, rest, st)) != cudaSuccess) return e;
        }
    }
    return cudaSuccess;
}

template <int E>
bool chain_serves_sim_e(int W, int cap, int K, int smem_max)
{
    ChPlan p;
    return ch_plan<E>(W, cap, K, smem_max, true, true, false, &p);
}

}  // namespace aladdin
