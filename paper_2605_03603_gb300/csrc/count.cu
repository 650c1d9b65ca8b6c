// Counting kernels: Algorithm 2 (BBVP, vertex-based pruning, Section 4.3) on
// the device.
//
// Notation. The anchor side X plays S of Algorithm 2; its vertices are
// renumbered by rank in the vertex priority rho (Definition 4). k is the tuple
// size on X and l the size on the other side Y (k = p, l = q when X = U;
// k = q, l = p when X = V); R = k - 1 partners join each anchor.
//
// Per anchor u (rank r):
//   position j of u's list Gamma(u) = (v_0, v_1, ...) is "useful" when the
//   suffix of v_j's list above r holds at least R entries: only then can v_j
//   be a common neighbour of u and R partners of higher rank. Useful
//   positions are numbered 0..d'-1 and become bit positions.
//   2-hop step (Algorithm 2, cnt and L maps): for every useful position j and
//   every w in the suffix of v_j: cnt[w] += 1, P_w[j] = 1 and
//   D_w[j] = (sign(u,v_j) != sign(w,v_j)). P_w is L[w] as a bitmask over
//   Gamma(u); D_w holds the type letter of Section 4.2 (set = d, clear = s).
//   Candidate filter (Algorithm 2): C = { w : cnt[w] >= l }.
//   Tuple step: every R-subset A of C with T = AND of P_w over A (nested
//   pruning: a prefix whose T already has fewer than l bits is dropped, which
//   drops only subsets with |T| < l). The type of v_j is the vector of D_w[j]
//   over A; x[type] = popc(T AND the matching D / NOT D masks), and the
//   anchor adds sum over types of binom(x[type], l).
// Positions that are not useful can never be in T, so leaving them out of
// cnt changes no term of the sum; the paper's own candidate set (counted
// over all positions) is also computed on request to report the number of
// subsets Algorithm 2 enumerates.
#include <algorithm>
#include <vector>

#include <cfloat>
#include <cstring>

#include "sbc_internal.cuh"

namespace sbc {

namespace {

constexpr uint32_t VMASK = 0x7FFFFFFFu;
constexpr uint32_t EMPTY = 0xFFFFFFFFu;
constexpr unsigned FULL = 0xFFFFFFFFu;

// ------------------------------------------------------------------ counters

// Device-side scalars of one count. Fields up to `run_begin` are set while
// planning (they stay valid when the counting kernels are replayed); the
// rest are accumulators and queue heads of one execution.
struct Counters {
    unsigned long long tuples_paper[2];// u128, sum binom(|C_paper|, R)
    unsigned long long tuples_ours[2]; // u128, sum binom(|C'|, R)
    unsigned long long candidates;     // sum |C'| (or |C_paper| in stats mode)
    unsigned long long e_max;          // largest visited-wedge count of a large anchor
    unsigned long long words_big, words_small;  // pool words of the two 2-hop tiers
    unsigned int n_active;             // anchors with work
    unsigned int n_direct;             // anchors for the direct 2-hop kernel,
    unsigned int n_big;                // ... for it and the CTA-wide hash kernel
    // tuple step of one anchor group
    double cost_total;                 // cost estimate of the work items
    unsigned int n_items;
    unsigned int n_warp;               // anchors counted one per warp
    unsigned int n_tc;                 // anchors for the tensor-core pair step
    unsigned int n_claims;             // anchors shared by several work items
    // ---- per execution
    unsigned long long run_begin;      // marker (unused)
    unsigned long long total[2];       // u128 count
    unsigned long long wedges;         // 2-hop entries visited
    unsigned long long tested;         // tuples whose common-neighbour mask was tested
    unsigned long long leaves;         // tuples with |T| >= l (type counts taken)
    unsigned long long popc_words;     // mask words popcounted by the tuple kernel and the self-checks
    // CTA-wide 2-hop kernel, by strategy (one window, bucketed, re-read windows,
    // bucketed with a second scatter)
    unsigned long long tw_reads;       // 2-hop entries read, all passes
    unsigned long long tw_cyc[4];      // SM cycles spent on its anchors
    unsigned long long tw_anchors[4];
    unsigned long long tw_fin_max, tw_fin_min_n;  // CTA finish times (global ns; min kept as ~t)
    unsigned long long tw_split;       // hash classes hashed in sub-class windows
    unsigned int head_direct;          // 2-hop queue heads
    unsigned int head_large;
    unsigned int head_small;
    unsigned int head_b;               // tuple queue heads: work items,
    unsigned int head_w;               // ... small anchors
    unsigned int err;                  // error bits
};

enum : unsigned {
    CERR_OVERFLOW = kErrOverflow,  // a binomial or the sum left 128 bits
    CERR_TIMEOUT = kErrTimeout,    // a bounded wait of the tensor-core kernel ran out
    CERR_RESERVE = 2u,    // candidate reservation exceeded (cannot happen)
    CERR_HASH = 4u,       // 2-hop table overflow after all retries
    CERR_MASK = 8u,       // self-check: a candidate mask disagrees with its 2-hop counters
};

// Thresholds: the largest x for which binom(x, l) is computed exactly in 64
// bits by the multiplicative formula (index l, 0..8).
__constant__ unsigned long long c_binom64_max[9];

// ------------------------------------------------------------------ binomials

__device__ __forceinline__ void div_u128_small(unsigned long long &lo, unsigned long long &hi,
                                               unsigned d) {
    unsigned long long qh = hi / d;
    unsigned long long r = hi % d;
    unsigned long long a = (r << 32) | (lo >> 32);
    unsigned long long q1 = a / d;
    r = a % d;
    unsigned long long b = (r << 32) | (lo & 0xFFFFFFFFull);
    unsigned long long q0 = b / d;
    hi = qh;
    lo = (q1 << 32) | q0;
}

// (lo, hi) *= m; returns false on 128-bit overflow.
__device__ __forceinline__ bool mul_u128_u64(unsigned long long &lo, unsigned long long &hi,
                                             unsigned long long m) {
    unsigned long long l0 = lo * m;
    unsigned long long c = __umul64hi(lo, m);
    unsigned long long h0 = hi * m;
    unsigned long long hh = __umul64hi(hi, m);
    unsigned long long nh = h0 + c;
    bool ovf = hh != 0 || nh < h0;
    lo = l0;
    hi = nh;
    return !ovf;
}

__device__ __forceinline__ unsigned gcd_u32(unsigned a, unsigned b) {
    while (b) {
        unsigned t = a % b;
        a = b;
        b = t;
    }
    return a;
}

template <int L>
__device__ __forceinline__ unsigned long long binom_u64(unsigned long long x) {
    unsigned long long r = 1;
#pragma unroll
    for (int i = 1; i <= L; i++) r = r * (x - L + i) / (unsigned long long)i;
    return r;
}

// binom(x, l) in 128 bits, exact (returned by value so that callers'
// accumulators stay in registers). Sets CERR_OVERFLOW if it needs more.
__device__ __noinline__ U128 binom_slow(unsigned long long x, int l, unsigned *err) {
    U128 t;
    unsigned long long lo = 1, hi = 0;
    for (int i = 1; i <= l; i++) {
        unsigned long long f = x - l + i;
        unsigned g = gcd_u32((unsigned)(f % (unsigned)i), (unsigned)i);
        if (g == 0) g = (unsigned)i;
        div_u128_small(lo, hi, (unsigned)i / g);
        if (!mul_u128_u64(lo, hi, f / g)) {
            atomicOr(err, CERR_OVERFLOW);
            return t;
        }
    }
    t.lo = lo;
    t.hi = hi;
    return t;
}

__device__ __forceinline__ void binom_add(U128 &acc, unsigned x, int l, unsigned *err) {
    if ((int)x < l) return;
    if (x > c_binom64_max[l]) {
        if (acc.add(binom_slow(x, l, err))) atomicOr(err, CERR_OVERFLOW);
        return;
    }
    unsigned long long v;
    switch (l) {
        case 2: v = binom_u64<2>(x); break;
        case 3: v = binom_u64<3>(x); break;
        case 4: v = binom_u64<4>(x); break;
        case 5: v = binom_u64<5>(x); break;
        case 6: v = binom_u64<6>(x); break;
        case 7: v = binom_u64<7>(x); break;
        default: v = binom_u64<8>(x); break;
    }
    acc.add(v);
}

// ---- direct 2-hop counters. A partner's rank follows the anchor's, and anchors with
// many wedges have high degrees, so high ranks: their partners' ranks span a
// short range (on the 2M-edge graph 76 % of the wedges of anchors above 3,584
// span at most 48k ranks). Such an anchor counts its partners in a table
// indexed by rank - no keys, no probes, one shared-memory add without a return
// value per wedge - in windows of consecutive ranks, each a pass over the
// 2-hop. Counters hold the same-sign and different-sign counts of a partner in
// 8 + 8 bits (at most 255 useful positions) or 16 + 16 bits. After a window's
// counts, a bitmap of the parts with at least l positions and its prefix counts
// number the rows, and the counters' memory stages the mask words of the
// window's rows, a range of positions at a time.
// Bound by the latency of the gathers of B_ent, four in flight per lane, and by
// the barriers between an anchor's passes (stalls per issue 8.0 and 6.4; LSU pipe
// 22 %, L2 20 % on the 500k-edge graph). The 2-hop kernels of the (3,3) count
// took 13.7 -> 4.9 ms on the 2M-edge graph, 79 -> 23 ms on a 12M-edge hub
// graph and 15.6 -> 1.0 ms on a dense 3000 x 800 graph
// (hash strategies -> direct counters where the rule takes them).
constexpr int DT_THREADS = 512;
constexpr int DT_WARPS = DT_THREADS / 32;
constexpr int DT_PCH = DT_THREADS;               // positions staged at once
constexpr uint32_t DT_WORDS = 20480;            // counter words, then staged mask words
constexpr uint32_t DT_CELLS8 = 2 * DT_WORDS;    // ranks per window with 8 + 8 bit counters
constexpr uint32_t DT_CELLS16 = DT_WORDS;
constexpr uint32_t DT_BM = DT_CELLS8 / 16;      // bitmap words (two bits per rank)
constexpr size_t DT_OFF_BM = (size_t)DT_WORDS * 4;
constexpr size_t DT_OFF_PRE = DT_OFF_BM + (size_t)DT_BM * 4;
constexpr size_t DT_OFF_POFF = DT_OFF_PRE + (size_t)DT_BM * 4;
constexpr size_t DT_OFF_PPRE = DT_OFF_POFF + (size_t)DT_PCH * 4;
constexpr size_t DT_OFF_PINFO = DT_OFF_PPRE + (size_t)(DT_PCH + 4) * 4;
constexpr size_t DT_SMEM = DT_OFF_PINFO + (size_t)DT_PCH * 4;

// Direct counters or the hash strategies. Lists of at least 8 partners on
// average (in shorter ones, of the widest hubs, few partners share all the
// counters). Costs in SM cycles measured on the 2M-edge graph: a window about
// 3,000 (clear, scan, barriers) and 0.7 per wedge for its two passes; the hash
// strategies about 8 per wedge.
__device__ __forceinline__ bool direct_takes(unsigned long long e, uint32_t dp, uint32_t range) {
    if (dp > 65535u || e < 8ull * dp) return false;
    const uint32_t cells = dp <= 255u ? DT_CELLS8 : DT_CELLS16;
    const float nwin = (float)((range + cells - 1) / cells);
    return nwin * (3000.0f + 0.7f * (float)e) < 8.0f * (float)e;
}

// ------------------------------------------------------------------ plan

struct PlanArgs {
    const int64_t *A_off;
    const uint32_t *A_ent, *A_pos;
    const int64_t *B_off;
    int64_t nX;
    int64_t chunks;            // of rows (k_plan): at least nX / PLAN_ROWS
    int R, l, shard, nshard, stats, small_e;
    int direct;                // direct counters allowed (not when a test forces the hash strategies)
    const int64_t *graph_x0;   // batches: first rank per graph (n_graphs + 1), else null
    int n_graphs;
    uint32_t *A_bit, *dprime, *rsv_c;
    unsigned long long *e_use, *e_all;  // e_all: with stats only
    uint8_t *key;
    uint32_t *hist;  // anchors per key
    Counters *cnt;
};

// One past the last rank that anchor r's partners can have: the side's, in a
// batch its own graph's.
__device__ __forceinline__ uint32_t rank_end(const int64_t *graph_x0, int n_graphs, uint32_t n_ranks, uint32_t r) {
    if (!graph_x0) return n_ranks;
    int lo = 0, hi = n_graphs;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (graph_x0[mid] <= (int64_t)r) lo = mid; else hi = mid;
    }
    return (uint32_t)graph_x0[lo + 1];
}

// Order key of an anchor, heavy first: 0..63 for the direct 2-hop tier, 64..127
// for the CTA-wide hash tier (two steps per octave of visited wedges), 128..254
// for the warp tier (four), 255 without work. The order only balances the work,
// so one pass over 256 keys is enough (four radix passes over 32-bit costs were
// a third of a small count's launches).
enum : int { TIER_DIRECT = 0, TIER_LARGE = 1, TIER_SMALL = 2 };
__device__ __forceinline__ uint32_t plan_key(unsigned long long cost, int tier) {
    const uint32_t x = cost < 0xFFFFFFFFull ? (uint32_t)cost : 0xFFFFFFFFu;
    const uint32_t e = 31 - __clz(x | 1u);
    if (tier == TIER_SMALL) {
        const uint32_t q = 4 * e + (e >= 2 ? (x >> (e - 2)) & 3u : 0u);
        return 128u + (q < 126u ? 126u - q : 0u);
    }
    const uint32_t q = 2 * e + (e >= 1 ? (x >> (e - 1)) & 1u : 0u);  // 0..63
    return (tier == TIER_DIRECT ? 63u : 127u) - q;
}

// Useful positions, wedge counts, reservation and order key of every anchor.
// Eight lanes per row up to PLAN_GROUP entries, a warp up to PLAN_WARP, else the
// CTA (a hub's 29,000 positions on one warp were 0.9 ms of a 1 ms plan).
constexpr int PLAN_THREADS = 256, PLAN_WARPS = PLAN_THREADS / 32, PLAN_ROWS = 4 * PLAN_WARPS;
constexpr int64_t PLAN_GROUP = 64, PLAN_WARP = 1024;

__global__ void __launch_bounds__(PLAN_THREADS) k_plan(PlanArgs a) {
    __shared__ uint32_t s_hist[256];
    __shared__ uint32_t s_cnt[2][4 * PLAN_WARPS];
    __shared__ unsigned long long s_sum[4][PLAN_WARPS];
    __shared__ unsigned s_act[3];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    s_hist[tid] = 0;
    if (tid < 3) s_act[tid] = 0;
    __syncthreads();
    unsigned long long words_big = 0, words_small = 0, e_max = 0;
    unsigned n_act = 0, n_big = 0, n_direct = 0;
    // a row's results (one thread)
    auto finish = [&](int64_t r, int64_t d, uint32_t dp, unsigned long long eu, unsigned long long ea) {
        const bool mine = a.nshard <= 1 || (r % a.nshard) == a.shard;
        const unsigned long long least = (unsigned long long)a.R * a.l;
        const bool active = mine && (a.stats ? d >= a.l && ea >= least : dp >= (uint32_t)a.l && eu >= least);
        // rows (candidate parts with >= l positions) the masks need room for;
        // one partner needs none (its 2-hop counters are enough)
        unsigned long long rc = 0;
        if (active && a.R > 1) {
            rc = eu / (unsigned long long)a.l;  // each row owns >= l useful wedges
            const unsigned long long above = 2 * (unsigned long long)(a.nX - 1 - r);
            rc = rc < above ? rc : above;
        }
        a.dprime[r] = dp;
        a.e_use[r] = eu;
        if (a.stats) a.e_all[r] = ea;
        a.rsv_c[r] = (uint32_t)rc;
        uint32_t key = 255;
        if (active) {
            const unsigned long long cost = a.stats ? ea : eu, words = (dp + 31) / 32 * rc;
            const bool big = cost > (unsigned long long)a.small_e;
            const bool direct = big && a.direct && !a.stats &&
                                direct_takes(eu, dp, rank_end(a.graph_x0, a.n_graphs, (uint32_t)a.nX, (uint32_t)r) -
                                                         1 - (uint32_t)r);
            key = plan_key(cost, direct ? TIER_DIRECT : big ? TIER_LARGE : TIER_SMALL);
            n_act++;
            n_direct += direct;
            if (big) {
                n_big++;
                words_big += words;
                e_max = cost > e_max ? cost : e_max;
            } else {
                words_small += words;
            }
            atomicAdd(&s_hist[key], 1u);
        }
        a.key[r] = (uint8_t)key;
    };
    auto suffix = [&](int64_t e) -> unsigned long long {
        const uint32_t y = a.A_ent[e] & VMASK;
        return (unsigned long long)(a.B_off[y + 1] - a.B_off[y] - (int64_t)a.A_pos[e] - 1);
    };
    // The rows of a step are chunks apart: the hubs, which rank next to one
    // another, go to different CTAs (32 of them on one were 1.1 ms)
    const int64_t chunks = a.chunks;
    for (int64_t ch = blockIdx.x; ch < chunks; ch += gridDim.x) {
        // four rows per warp, eight lanes each
        const int64_t r = ch + chunks * (4 * warp + (lane >> 3));
        int64_t e0 = 0, d = 0;
        if (r < a.nX) {
            e0 = a.A_off[r];
            d = a.A_off[r + 1] - e0;
        }
        const bool grouped = r < a.nX && d <= PLAN_GROUP;
        const uint32_t sub = lane & 7, sh = lane & 24;
        uint32_t dp = 0;
        unsigned long long eu = 0, ea = 0;
        const uint32_t steps = __reduce_max_sync(FULL, grouped ? (uint32_t)((d + 7) / 8) : 0u);
        for (uint32_t t = 0; t < steps; t++) {
            const int64_t k = 8 * (int64_t)t + sub;
            const bool in = grouped && k < d;
            const unsigned long long suf = in ? suffix(e0 + k) : 0ull;
            const bool useful = in && suf >= (unsigned long long)a.R;
            const uint32_t bal = (__ballot_sync(FULL, useful) >> sh) & 0xFFu;
            if (in) a.A_bit[e0 + k] = useful ? dp + __popc(bal & ((1u << sub) - 1u)) : EMPTY;
            dp += __popc(bal);
            eu += useful ? suf : 0ull;
            ea += suf;
        }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) {
            eu += __shfl_xor_sync(FULL, eu, o);
            ea += __shfl_xor_sync(FULL, ea, o);
        }
        if (grouped && sub == 0) finish(r, d, dp, eu, ea);
        // longer rows of the warp's four, one at a time
        for (uint32_t todo = __ballot_sync(FULL, sub == 0 && r < a.nX && d > PLAN_GROUP && d <= PLAN_WARP); todo;
             todo &= todo - 1) {
            const int src = __ffs(todo) - 1;
            const int64_t rr = __shfl_sync(FULL, r, src), f0 = __shfl_sync(FULL, e0, src),
                          dd = __shfl_sync(FULL, d, src);
            uint32_t p = 0;
            unsigned long long su = 0, sa = 0;
            for (int64_t k0 = 0; k0 < dd; k0 += 32) {
                const int64_t k = k0 + lane;
                const bool in = k < dd;
                const unsigned long long suf = in ? suffix(f0 + k) : 0ull;
                const bool useful = in && suf >= (unsigned long long)a.R;
                const uint32_t bal = __ballot_sync(FULL, useful);
                if (in) a.A_bit[f0 + k] = useful ? p + __popc(bal & ((1u << lane) - 1u)) : EMPTY;
                p += __popc(bal);
                su += useful ? suf : 0ull;
                sa += suf;
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                su += __shfl_xor_sync(FULL, su, o);
                sa += __shfl_xor_sync(FULL, sa, o);
            }
            if (lane == 0) finish(rr, dd, p, su, sa);
        }
        // the longest rows, by the CTA, four entries per thread and step
        if (!__syncthreads_or(sub == 0 && r < a.nX && d > PLAN_WARP)) continue;
        for (int64_t rr = ch; rr < a.nX; rr += chunks) {
            const int64_t f0 = a.A_off[rr], dd = a.A_off[rr + 1] - f0;
            if (dd <= PLAN_WARP) continue;
            uint32_t p = 0;
            unsigned long long su = 0, sa = 0;
            int flip = 0;
            for (int64_t k0 = 0; k0 < dd; k0 += 4 * PLAN_THREADS, flip ^= 1) {
                unsigned long long suf[4];
                uint32_t bal[4];
#pragma unroll
                for (int q = 0; q < 4; q++) {
                    const int64_t k = k0 + q * PLAN_THREADS + tid;
                    suf[q] = k < dd ? suffix(f0 + k) : 0ull;
                }
#pragma unroll
                for (int q = 0; q < 4; q++) {
                    bal[q] = __ballot_sync(FULL, suf[q] >= (unsigned long long)a.R && k0 + q * PLAN_THREADS + tid < dd);
                    if (lane == 0) s_cnt[flip][q * PLAN_WARPS + warp] = __popc(bal[q]);
                }
                __syncthreads();
                // (the other half of s_cnt is written in the next step)
                const uint32_t x = s_cnt[flip][lane];
                uint32_t incl = x;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t t = __shfl_up_sync(FULL, incl, o);
                    if (lane >= o) incl += t;
                }
#pragma unroll
                for (int q = 0; q < 4; q++) {
                    const uint32_t pre = __shfl_sync(FULL, incl - x, q * PLAN_WARPS + warp);
                    const int64_t k = k0 + q * PLAN_THREADS + tid;
                    if (k < dd) {
                        const bool useful = (bal[q] >> lane) & 1u;
                        a.A_bit[f0 + k] = useful ? p + pre + __popc(bal[q] & ((1u << lane) - 1u)) : EMPTY;
                        su += useful ? suf[q] : 0ull;
                        sa += suf[q];
                    }
                }
                p += __shfl_sync(FULL, incl, 31);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                su += __shfl_xor_sync(FULL, su, o);
                sa += __shfl_xor_sync(FULL, sa, o);
            }
            __syncthreads();
            if (lane == 0) {
                s_sum[0][warp] = su;
                s_sum[1][warp] = sa;
            }
            __syncthreads();
            if (tid == 0) {
                su = sa = 0;
                for (int w = 0; w < PLAN_WARPS; w++) {
                    su += s_sum[0][w];
                    sa += s_sum[1][w];
                }
                finish(rr, dd, p, su, sa);
            }
            __syncthreads();
        }
    }
    // the CTA's totals
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        words_big += __shfl_xor_sync(FULL, words_big, o);
        words_small += __shfl_xor_sync(FULL, words_small, o);
        const unsigned long long t = __shfl_xor_sync(FULL, e_max, o);
        e_max = t > e_max ? t : e_max;
    }
    n_act = __reduce_add_sync(FULL, n_act);
    n_big = __reduce_add_sync(FULL, n_big);
    n_direct = __reduce_add_sync(FULL, n_direct);
    __syncthreads();
    if (lane == 0) {
        s_sum[0][warp] = words_big;
        s_sum[1][warp] = words_small;
        s_sum[2][warp] = e_max;
        if (n_act) atomicAdd(&s_act[0], n_act);
        if (n_big) atomicAdd(&s_act[1], n_big);
        if (n_direct) atomicAdd(&s_act[2], n_direct);
    }
    __syncthreads();
    if (s_hist[tid]) atomicAdd(&a.hist[tid], s_hist[tid]);
    if (tid == 0 && s_act[0]) {
        for (int w = 1; w < PLAN_WARPS; w++) {
            words_big += s_sum[0][w];
            words_small += s_sum[1][w];
            e_max = s_sum[2][w] > e_max ? s_sum[2][w] : e_max;
        }
        atomicAdd(&a.cnt->n_active, s_act[0]);
        if (words_small) atomicAdd(&a.cnt->words_small, words_small);
        if (s_act[1]) {
            atomicAdd(&a.cnt->n_big, s_act[1]);
            if (s_act[2]) atomicAdd(&a.cnt->n_direct, s_act[2]);
            atomicAdd(&a.cnt->words_big, words_big);
            atomicMax(&a.cnt->e_max, e_max);
        }
    }
}

// Order of the active anchors by key (in any order within one), and their pool
// offsets when all fit one group: the CTA-wide tier's regions first, then the
// warp tier's. cursor: anchors placed per key, then the words placed per tier.
__global__ void __launch_bounds__(256) k_order(const uint8_t *__restrict__ key, int64_t nX,
                                               const uint32_t *__restrict__ hist,
                                               const uint32_t *__restrict__ dprime,
                                               const uint32_t *__restrict__ rsv_c, uint32_t *cursor,
                                               unsigned long long *word_cursor, const Counters *cnt,
                                               uint32_t *order, int64_t *pool_off) {
    __shared__ uint32_t s_base[256], s_tot[8];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    {
        const uint32_t x = tid < 255 ? hist[tid] : 0u;
        uint32_t incl = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(FULL, incl, o);
            if (lane >= o) incl += t;
        }
        if (lane == 31) s_tot[warp] = incl;
        __syncthreads();
        uint32_t pre = 0;
        for (int w = 0; w < warp; w++) pre += s_tot[w];
        s_base[tid] = pre + incl - x;
        __syncthreads();
    }
    const unsigned long long small0 = cnt->words_big;
    const uint32_t lt = (1u << lane) - 1u;
    for (int64_t r0 = blockIdx.x * 256ll; r0 < nX; r0 += gridDim.x * 256ll) {
        const int64_t r = r0 + tid;
        const uint32_t k = r < nX ? key[r] : 255u;
        const bool on = k != 255u;
        const uint32_t peers = __match_any_sync(FULL, k);
        uint32_t at = 0;
        if (on && (peers & lt) == 0) at = s_base[k] + atomicAdd(&cursor[k], (uint32_t)__popc(peers));
        at = __shfl_sync(FULL, at, __ffs(peers) - 1);
        if (on) order[at + __popc(peers & lt)] = (uint32_t)r;
        // pool words of the warp's anchors of each tier
        const bool big = k < 128u;
        const unsigned long long words = on ? (unsigned long long)((dprime[r] + 31) / 32) * rsv_c[r] : 0ull;
        unsigned long long wb = big ? words : 0ull, ws = big ? 0ull : words;
        const unsigned long long mb = wb, ms = ws;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long t = __shfl_up_sync(FULL, wb, o), u = __shfl_up_sync(FULL, ws, o);
            if (lane >= o) {
                wb += t;
                ws += u;
            }
        }
        unsigned long long ob = 0, os = 0;
        if (lane == 31) {
            if (wb) ob = atomicAdd(&word_cursor[0], wb);
            if (ws) os = atomicAdd(&word_cursor[1], ws);
        }
        ob = __shfl_sync(FULL, ob, 31);
        os = __shfl_sync(FULL, os, 31);
        if (on) pool_off[r] = (int64_t)(big ? ob + wb - mb : small0 + os + ws - ms);
    }
}

// ------------------------------------------------------------------ 2-hop

// Hash value: three 21-bit counters of one 2-hop partner w of the anchor.
//   bits  0..20  cnt over all positions (Algorithm 2's cnt[w])
//   bits 21..41  cnt over useful positions (|P_w|)
//   bits 42..62  useful positions with sign(u,v) != sign(w,v) (|D_w|)
//   bit  63      set once w is kept; bits 0..20 then hold its first row's index
//                (the other two counters stay: they tell its parts, and the
//                mask self-check uses them)
constexpr unsigned long long F_ALL = 1ull, F_USE = 1ull << 21, F_DIFF = 1ull << 42;
constexpr unsigned long long M21 = (1ull << 21) - 1;
constexpr unsigned long long CAND = 1ull << 63;
constexpr uint32_t NOBIT = 0x7FFFFFFFu;

__device__ __forceinline__ uint32_t hash_slot(uint32_t w, uint32_t hs) {
    return __umulhi(w * 0x9E3779B1u, hs);
}
__device__ __forceinline__ uint32_t class_mix(uint32_t w) {
    return ((w * 0x85EBCA6Bu) ^ (w >> 15)) * 0xC2B2AE35u;
}
// Hash class of w among 2^lg (the top lg bits of its mix) ...
__device__ __forceinline__ uint32_t class_of(uint32_t w, int lg) {
    return lg ? class_mix(w) >> (32 - lg) : 0u;
}
// ... and its sub-class among 2^lg2 within that class (the next lg2 bits).
__device__ __forceinline__ uint32_t subclass_of(uint32_t w, int lg, int lg2) {
    return lg2 ? (class_mix(w) << lg) >> (32 - lg2) : 0u;
}

// Add `add` to w's counters (open addressing, linear probing, at most hs
// probes). Returns false when the table is full.
__device__ __forceinline__ bool tab_insert(uint32_t *keys, unsigned long long *vals, uint32_t hs,
                                           uint32_t w, unsigned long long add) {
    uint32_t sl = hash_slot(w, hs);
    for (uint32_t probes = 0; probes < hs; probes++) {
        uint32_t k = keys[sl];
        if (k == EMPTY) {
            uint32_t old = atomicCAS(&keys[sl], EMPTY, w);
            if (old == EMPTY || old == w) {
                atomicAdd(&vals[sl], add);
                return true;
            }
            k = old;
        }
        if (k == w) {
            atomicAdd(&vals[sl], add);
            return true;
        }
        sl = (sl + 1 == hs) ? 0u : sl + 1;
    }
    return false;
}

__device__ __forceinline__ int tab_find(const uint32_t *keys, uint32_t hs, uint32_t w) {
    uint32_t sl = hash_slot(w, hs);
    for (uint32_t probes = 0; probes < hs; probes++) {
        uint32_t k = keys[sl];
        if (k == w) return (int)sl;
        if (k == EMPTY) return -1;
        sl = (sl + 1 == hs) ? 0u : sl + 1;
    }
    return -1;
}

// Candidate filter. Algorithm 2 keeps w when cnt[w] >= l. Every type class
// of a tuple through w lies inside the same-sign or the different-sign part
// of L[w] (the letter c_w is constant on a class), so only parts with at least
// l useful common neighbours can add a non-zero binomial: each of them becomes
// a row of mask words, the others are dropped, which changes no term.
__device__ __forceinline__ uint32_t use_count(unsigned long long v) { return (uint32_t)((v >> 21) & M21); }
__device__ __forceinline__ uint32_t diff_count(unsigned long long v) { return (uint32_t)((v >> 42) & M21); }
__device__ __forceinline__ bool keep_same(unsigned long long v, int l) {
    return use_count(v) - diff_count(v) >= (uint32_t)l;
}
__device__ __forceinline__ bool keep_diff(unsigned long long v, int l) { return diff_count(v) >= (uint32_t)l; }

__device__ __forceinline__ unsigned long long pass1_add(uint32_t sdiff, uint32_t bit) {
    return bit != EMPTY ? (F_ALL | F_USE | (sdiff ? F_DIFF : 0ull)) : F_ALL;
}

// Kept candidate: its first row's index in bits 0..20 (same-sign part first),
// the two useful-position counters kept, CAND set.
__device__ __forceinline__ unsigned long long cand_value(unsigned long long v, uint32_t row) {
    return CAND | (v & ~(CAND | M21)) | (unsigned long long)row;
}
// Row of the part `sdiff` of a kept candidate, EMPTY when that part was dropped.
__device__ __forceinline__ uint32_t row_index(unsigned long long v, uint32_t sdiff, int l) {
    const uint32_t base = (uint32_t)(v & M21);
    const bool same = keep_same(v, l);
    if (!sdiff) return same ? base : EMPTY;
    return keep_diff(v, l) ? base + (same ? 1u : 0u) : EMPTY;
}

// Self-check of one row after its mask is written: its popcount must equal
// the positions its counter holds. Consecutive words are `stride` apart. Reads
// of global rows bypass L1 (the words were written by atomics at L2).
__device__ __forceinline__ bool row_matches(const uint32_t *row, size_t stride, uint32_t W, uint32_t want,
                                            bool global) {
    uint32_t n = 0;
    for (uint32_t w = 0; w < W; w++) n += __popc(global ? __ldcg(row + w * stride) : row[w * stride]);
    return n == want;
}
__device__ __forceinline__ bool rows_match(const uint32_t *rows, size_t stride, uint32_t W,
                                           unsigned long long v, int l, bool global, unsigned long long &words) {
    const uint32_t s = row_index(v, 0, l), d = row_index(v, 1, l);
    words += (unsigned long long)W * ((s != EMPTY) + (d != EMPTY));
    return (s == EMPTY || row_matches(rows + s, stride, W, use_count(v) - diff_count(v), global)) &&
           (d == EMPTY || row_matches(rows + d, stride, W, diff_count(v), global));
}

// Where a count's sums go: the total, and per anchor or per graph of a batch.
struct Totals {
    unsigned long long *total;       // u128
    unsigned long long *per_anchor;  // u128 per anchor rank, or null
    unsigned long long *per_graph;   // u128 per graph of a batch, or null
    const int64_t *graph_x0;         // first anchor rank of each graph (n_graphs + 1)
    int n_graphs;
    unsigned *err;
};

// Add one anchor's (partial) sum; called by one lane.
__device__ __forceinline__ void add_totals(const Totals &t, uint32_t r, const U128 &s) {
    if (!(s.lo | s.hi)) return;
    // a batch's union total is not a count (its graphs' totals are)
    atomic_add_u128(t.total, s.lo, s.hi, t.per_graph ? nullptr : t.err);
    if (t.per_anchor) atomic_add_u128(t.per_anchor + 2 * (size_t)r, s.lo, s.hi, t.err);
    if (t.per_graph) {
        int lo = 0, hi = t.n_graphs;  // largest g with graph_x0[g] <= r
        while (hi - lo > 1) {
            int mid = (lo + hi) >> 1;
            if (t.graph_x0[mid] <= (int64_t)r) lo = mid; else hi = mid;
        }
        atomic_add_u128(t.per_graph + 2 * (size_t)lo, s.lo, s.hi, t.err);
    }
}

// What the tuple step's plan wants to know about an anchor's rows: positions
// of all of them, and of the longest (after it: the plan, see AnchorPlan).
struct RowInfo {
    float pops = 0;
    uint32_t longest = 0;
    __device__ __forceinline__ void add(uint32_t pop) {
        pops += (float)pop;
        longest = pop > longest ? pop : longest;
    }
    __device__ __forceinline__ void warp_sum() {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) pops += __shfl_xor_sync(FULL, pops, o);
        longest = __reduce_max_sync(FULL, longest);
    }
};

struct TwohopArgs {
    const int64_t *A_off;
    const uint32_t *A_ent, *A_pos, *A_bit;
    const int64_t *B_off;
    const uint32_t *B_ent;
    const uint32_t *dprime;
    const unsigned long long *e_use, *e_all;
    const uint32_t *rsv_c;
    const int64_t *pool_off;
    const uint32_t *order;
    uint32_t *pool;
    uint32_t *ncand, *npaper, *nrow;
    RowInfo *rinfo;
    Counters *cnt;
    Totals tot;
    uint32_t n_ranks;               // anchors of the side
    int single;                     // one partner: the counters give the sum, no rows are written
    unsigned long long *bucket;     // per-CTA bucket slots of the large-anchor kernel
    unsigned long long bucket_slot; // entries per slot
    unsigned direct_begin, direct_end;  // order[] ranges of the three kernels
    unsigned large_begin, large_end;
    unsigned small_begin, small_end;
    int l;
    int check;                      // run the candidate-mask self-check
    uint32_t hs_cap;                // test override: most hash slots per table (0: none)
    uint32_t wcap;                  // most visited wedges of a one-window anchor
};

// Table size after the test override (which makes tables overflow on purpose,
// to drive the CERR_HASH path).
__device__ __forceinline__ uint32_t cap_slots(uint32_t hs, const TwohopArgs &a) {
    return (a.hs_cap && hs > a.hs_cap) ? a.hs_cap : hs;
}

// ---- small anchors: one warp per anchor, private table in shared memory

constexpr int PS_THREADS = 256;
constexpr int PS_WARPS = PS_THREADS / 32;
constexpr int PS_HS = 1024;            // slots per warp
// Default and largest tier threshold in visited wedges (table load <= 1/2).
constexpr int SMALL_E_MAX = PS_HS / 2;
constexpr size_t PS_SMEM = (size_t)PS_WARPS * PS_HS * 12;

// Visit the anchor's 2-hop entries with one warp. fn(w, sdiff, bit).
template <typename F>
__device__ __forceinline__ void visit_warp(int64_t ebase, int d, bool useful_only,
                                           const uint32_t *__restrict__ A_ent,
                                           const uint32_t *__restrict__ A_pos,
                                           const uint32_t *__restrict__ A_bit,
                                           const int64_t *__restrict__ B_off,
                                           const uint32_t *__restrict__ B_ent, F fn) {
    const int lane = threadIdx.x & 31;
    for (int g = 0; g < d; g += 32) {
        int j = g + lane;
        int64_t start = 0;
        uint32_t len = 0, su = 0, bit = EMPTY;
        if (j < d) {
            int64_t e = ebase + j;
            uint32_t av = A_ent[e];
            uint32_t y = av & VMASK;
            su = av >> 31;
            bit = A_bit[e];
            start = B_off[y] + (int64_t)A_pos[e] + 1;
            len = (uint32_t)(B_off[y + 1] - start);
            if (useful_only && bit == EMPTY) len = 0;
        }
        uint32_t incl = len;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            uint32_t t = __shfl_up_sync(FULL, incl, o);
            if (lane >= o) incl += t;
        }
        uint32_t total = __shfl_sync(FULL, incl, 31);
        uint32_t excl = incl - len;
        for (uint32_t base = 0; base < total; base += 32) {
            uint32_t idx = base + lane;
            int s = 0;
#pragma unroll
            for (int step = 16; step > 0; step >>= 1) {
                uint32_t ex = __shfl_sync(FULL, excl, s + step);
                if (ex <= idx) s += step;
            }
            long long st = __shfl_sync(FULL, (long long)start, s);
            uint32_t exs = __shfl_sync(FULL, excl, s);
            uint32_t sus = __shfl_sync(FULL, su, s);
            uint32_t bits = __shfl_sync(FULL, bit, s);
            if (idx < total) {
                uint32_t ent = B_ent[st + (idx - exs)];
                fn(ent & VMASK, sus ^ (ent >> 31), bits);
            }
        }
    }
}

// The 2-hop kernels of one launch_twohop overlap: a kernel lets the next one start
// once all its CTAs run, and ends only after the one before it.
__device__ __forceinline__ void twohop_let_next_start() { asm volatile("griddepcontrol.launch_dependents;"); }
__device__ __forceinline__ void twohop_wait_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <bool STATS>
__global__ void __launch_bounds__(PS_THREADS) k_twohop_small(const __grid_constant__ TwohopArgs a) {
    twohop_let_next_start();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t *keys = (uint32_t *)(smem_raw + (size_t)warp * PS_HS * 4);
    unsigned long long *vals =
        (unsigned long long *)(smem_raw + (size_t)PS_WARPS * PS_HS * 4 + (size_t)warp * PS_HS * 8);
    const int l = a.l;
    const uint32_t lt = (1u << lane) - 1u;
    const bool split_totals = a.tot.per_anchor || a.tot.per_graph;
    unsigned long long wedges = 0, tested = 0, leaves = 0;
    U128 total;
    for (;;) {
        unsigned item = 0;
        if (lane == 0) item = atomicAdd(&a.cnt->head_small, 1u);
        item = __shfl_sync(FULL, item, 0) + a.small_begin;
        if (item >= a.small_end) break;
        const uint32_t r = a.order[item];
        const int64_t ebase = a.A_off[r];
        const int d = (int)(a.A_off[r + 1] - ebase);
        const uint32_t W = (a.dprime[r] + 31) / 32;
        const uint32_t rsv = a.rsv_c[r];
        uint32_t *region = a.pool + a.pool_off[r];
        const unsigned long long e_vis = STATS ? a.e_all[r] : a.e_use[r];
        uint32_t hs = (uint32_t)(2 * e_vis + 31) & ~31u;
        hs = hs < 64 ? 64 : (hs > PS_HS ? PS_HS : hs);
        hs = cap_slots(hs, a);
        for (uint32_t i = lane; i < hs; i += 32) {
            keys[i] = EMPTY;
            vals[i] = 0;
        }
        __syncwarp();
        bool ovf = false;
        visit_warp(ebase, d, !STATS, a.A_ent, a.A_pos, a.A_bit, a.B_off, a.B_ent,
                   [&](uint32_t w, uint32_t sdiff, uint32_t bit) {
                       if (!tab_insert(keys, vals, hs, w, pass1_add(sdiff, bit))) ovf = true;
                   });
        __syncwarp();
        uint32_t ncw = 0, nrow = 0, npaper = 0;
        RowInfo rst;
        U128 sum;
        if (__any_sync(FULL, ovf)) {
            if (lane == 0) atomicOr(&a.cnt->err, CERR_HASH);
        } else {
            for (uint32_t base = 0; base < hs; base += 32) {
                uint32_t i = base + lane;
                bool same = false, diff = false, pap = false;
                unsigned long long v = 0;
                if (i < hs && keys[i] != EMPTY) {
                    v = vals[i];
                    pap = STATS && (v & M21) >= (unsigned long long)l;
                    same = keep_same(v, l);
                    diff = keep_diff(v, l);
                }
                const uint32_t bs = __ballot_sync(FULL, same), bd = __ballot_sync(FULL, diff);
                if (same || diff) vals[i] = cand_value(v, nrow + __popc(bs & lt) + __popc(bd & lt));
                if (a.single) {
                    if (same) binom_add(sum, use_count(v) - diff_count(v), l, &a.cnt->err);
                    if (diff) binom_add(sum, diff_count(v), l, &a.cnt->err);
                } else {
                    if (same) rst.add(use_count(v) - diff_count(v));
                    if (diff) rst.add(diff_count(v));
                }
                ncw += __popc(bs | bd);
                nrow += __popc(bs) + __popc(bd);
                if (STATS) npaper += __popc(__ballot_sync(FULL, pap));
            }
            __syncwarp();
            if (a.single) {
                leaves += nrow;
                tested += ncw;
                if (nrow) {
                    const U128 ws = warp_sum_u128(sum, &a.cnt->err);
                    if (split_totals) {
                        if (lane == 0) add_totals(a.tot, r, ws);
                    } else if (total.add(ws)) {
                        atomicOr(&a.cnt->err, CERR_OVERFLOW);
                    }
                }
            } else if (nrow > rsv) {
                if (lane == 0) atomicOr(&a.cnt->err, CERR_RESERVE);
                ncw = nrow = 0;
            } else if (nrow > 0) {
                rst.warp_sum();
                // The small anchors' part of the pool is zeroed on the stream
                // before the 2-hop launches, so the rows are built by atomicOr
                // alone (no zeroing stores of this kernel ever meet its
                // atomics on the same words).
                visit_warp(ebase, d, true, a.A_ent, a.A_pos, a.A_bit, a.B_off, a.B_ent,
                           [&](uint32_t w, uint32_t sdiff, uint32_t bit) {
                               int sl = tab_find(keys, hs, w);
                               if (sl < 0) return;
                               unsigned long long v = vals[sl];
                               if (!(v & CAND)) return;
                               const uint32_t row = row_index(v, sdiff, l);
                               if (row != EMPTY)
                                   atomicOr(&region[(size_t)(bit >> 5) * rsv + row], 1u << (bit & 31));
                           });
                if (a.check) {
                    __syncwarp();
                    bool bad = false;
                    unsigned long long words = 0;
                    for (uint32_t i = lane; i < hs; i += 32) {
                        if (keys[i] == EMPTY) continue;
                        unsigned long long v = vals[i];
                        if ((v & CAND) && !rows_match(region, rsv, W, v, l, true, words)) bad = true;
                    }
                    if (words) atomicAdd(&a.cnt->popc_words, words);
                    if (__any_sync(FULL, bad) && lane == 0) atomicOr(&a.cnt->err, CERR_MASK);
                }
            }
        }
        if (lane == 0) {
            a.ncand[r] = ncw;
            a.nrow[r] = nrow;
            a.rinfo[r] = rst;
            if (STATS) a.npaper[r] = npaper;
        }
        wedges += e_vis;
        __syncwarp();
    }
    if (lane == 0) {
        add_totals(a.tot, 0, total);
        if (tested) atomicAdd(&a.cnt->tested, tested);
        if (leaves) atomicAdd(&a.cnt->leaves, leaves);
    }
    if (lane == 0 && wedges) atomicAdd(&a.cnt->wedges, wedges);
    twohop_wait_previous();
}

// ---- large anchors: one CTA per anchor, wedges flattened over the CTA

constexpr int PL_THREADS = 512;
constexpr int PL_WARPS = PL_THREADS / 32;
constexpr int PL_HS = 7168;             // slots
constexpr int PL_WCAP = PL_HS / 2;      // visited wedges per re-read window (load <= 1/2)
constexpr int PL_BCAP = PL_HS / 3;      // expected entries per bucket (bucket <= 1.5x + 64)
constexpr int PL_MAXCLS = 1024;         // bucket classes per anchor
constexpr int PL_PCH = PL_THREADS;      // positions staged per chunk
constexpr int PL_STAGE_WORDS = 4096;    // staged P/D words
constexpr size_t PL_OFF_VALS = (size_t)PL_HS * 4;
constexpr size_t PL_OFF_PST = PL_OFF_VALS + (size_t)PL_HS * 8;
constexpr size_t PL_OFF_PPRE = PL_OFF_PST + (size_t)PL_PCH * 8;
constexpr size_t PL_OFF_PINFO = PL_OFF_PPRE + (size_t)(PL_PCH + 4) * 4;
constexpr size_t PL_OFF_STAGE = PL_OFF_PINFO + (size_t)PL_PCH * 4;
constexpr size_t PL_SMEM = PL_OFF_STAGE + (size_t)PL_STAGE_WORDS * 4;

// Bucket entry of a wedge: w (bits 0..30), sdiff (bit 31), bit index of the
// position (bits 32..52; all ones when the position is not useful).
constexpr unsigned long long BE_NOBIT = (1ull << 21) - 1;

__device__ __forceinline__ unsigned long long bucket_entry(uint32_t w, uint32_t sdiff, uint32_t bit) {
    const unsigned long long bi = bit == EMPTY ? BE_NOBIT : (unsigned long long)bit;
    return (unsigned long long)w | ((unsigned long long)sdiff << 31) | (bi << 32);
}

__host__ __device__ __forceinline__ unsigned long long bucket_cap(unsigned long long e_vis, int lg) {
    return ((e_vis >> lg) * 3) / 2 + 65;
}

// Largest bucket area one anchor can need: sum of its classes' capacities.
__host__ __device__ __forceinline__ int bucket_lg(unsigned long long e_vis) {
    int lg = 0;
    while (((unsigned long long)PL_BCAP << lg) < e_vis && lg < 10) lg++;
    return lg;
}

__device__ __forceinline__ unsigned long long block_excl_scan_u64(unsigned long long v,
                                                                  unsigned long long *warp_tot,
                                                                  unsigned long long *total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int NW = PL_WARPS;
    unsigned long long incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        unsigned long long t = __shfl_up_sync(FULL, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) warp_tot[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        unsigned long long wv = lane < NW ? warp_tot[lane] : 0ull;
        unsigned long long wi = wv;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            unsigned long long t = __shfl_up_sync(FULL, wi, o);
            if (lane >= o) wi += t;
        }
        if (lane < NW) warp_tot[lane] = wi - wv;
        if (lane == NW - 1) *total = wi;
    }
    __syncthreads();
    return warp_tot[warp] + incl - v;
}

// Visit the anchor's 2-hop entries with the whole CTA; with lg_nw > 0 only
// entries of hash class `cls`. Positions are staged PL_PCH at a time and the
// non-empty ones compacted; each warp takes 32 consecutive entries, one
// binary search for the first and short forward walks for the others.
// fn(w, sdiff, bit).
template <typename F>
__device__ __forceinline__ void visit_block(int64_t ebase, int d, bool useful_only, int lg_nw,
                                            uint32_t cls, const TwohopArgs &a, int64_t *pst,
                                            uint32_t *ppre, uint32_t *pinfo,
                                            unsigned long long *warp_tot,
                                            unsigned long long *s_total, F fn) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int c0 = 0; c0 < d; c0 += PL_PCH) {
        const int nch = d - c0 < PL_PCH ? d - c0 : PL_PCH;
        uint32_t len = 0, info = 0;
        int64_t st = 0;
        if (tid < nch) {
            int64_t e = ebase + c0 + tid;
            uint32_t av = a.A_ent[e];
            uint32_t y = av & VMASK;
            uint32_t bit = a.A_bit[e];
            st = a.B_off[y] + (int64_t)a.A_pos[e] + 1;
            len = (uint32_t)(a.B_off[y + 1] - st);
            if (useful_only && bit == EMPTY) len = 0;
            info = (av & 0x80000000u) | (bit == EMPTY ? NOBIT : bit);
        }
        // scan of (non-empty flag, length): compact slot and entry prefix
        unsigned long long packed = len ? ((1ull << 32) | len) : 0ull;
        unsigned long long ex = block_excl_scan_u64(packed, warp_tot, s_total);
        if (len) {
            const uint32_t slot = (uint32_t)(ex >> 32);
            pst[slot] = st;
            pinfo[slot] = info;
            ppre[slot] = (uint32_t)ex;
        }
        __syncthreads();
        const uint32_t npos = (uint32_t)(*s_total >> 32);
        const uint32_t total = (uint32_t)*s_total;
        for (uint32_t base = (uint32_t)warp * 32; base < total; base += PL_THREADS) {
            uint32_t p0 = 0;
            if (lane == 0) {
                uint32_t lo = 0, hi = npos;  // largest j with ppre[j] <= base
                while (hi - lo > 1) {
                    uint32_t mid = (lo + hi) >> 1;
                    if (ppre[mid] <= base) lo = mid; else hi = mid;
                }
                p0 = lo;
            }
            uint32_t p = __shfl_sync(FULL, p0, 0);
            const uint32_t t = base + lane;
            if (t < total) {
                while (p + 1 < npos && ppre[p + 1] <= t) p++;
                uint32_t ent = a.B_ent[pst[p] + (t - ppre[p])];
                uint32_t w = ent & VMASK;
                if (lg_nw == 0 || class_of(w, lg_nw) == cls) {
                    uint32_t inf = pinfo[p];
                    uint32_t bit = inf & NOBIT;
                    fn(w, (inf >> 31) ^ (ent >> 31), bit == NOBIT ? EMPTY : bit);
                }
            }
        }
        __syncthreads();
    }
}

// ---- direct counters (see their description above the plan)

// Positions staged in shared memory: list p's entries t in [ppre[p], ppre[p + 1])
// are B_ent[poff[p] + t], pinfo[p] holds the sign of the position and its bit
// index.
struct Lists {
    uint32_t *poff, *ppre, *pinfo;
    uint32_t *wtot;  // DT_WARPS + 1 words: scan scratch
};

// Exclusive scan of one 32-bit value per thread over the CTA; *total: the sum.
__device__ __forceinline__ uint32_t block_excl_scan_u32(uint32_t v, uint32_t *wtot, uint32_t *total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(FULL, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) wtot[warp] = incl;
    __syncthreads();
    const uint32_t x = lane < DT_WARPS ? wtot[lane] : 0u;
    uint32_t xi = x;
#pragma unroll
    for (int o = 1; o < DT_WARPS; o <<= 1) {
        const uint32_t t = __shfl_up_sync(FULL, xi, o);
        if (lane >= o) xi += t;
    }
    *total = __shfl_sync(FULL, xi, DT_WARPS - 1);
    return __shfl_sync(FULL, xi - x, warp) + incl - v;
}

// Walk the entries of the staged lists [plo, phi) with the whole CTA: split
// evenly over the warps; every lane finds its first list by a search and walks
// forward from it, four entries in flight. fn(entry, sign | bit index).
template <typename F>
__device__ __forceinline__ void walk_lists(const Lists &L, uint32_t plo, uint32_t phi,
                                           const uint32_t *__restrict__ B_ent, F fn) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t tb = L.ppre[plo], te = L.ppre[phi];
    const uint32_t per = ((te - tb + DT_THREADS - 1) / DT_THREADS) * 32;
    const uint32_t t1 = min(te, tb + (uint32_t)(warp + 1) * per);
    uint32_t t = tb + (uint32_t)warp * per + lane;
    if (t >= t1) return;
    uint32_t p = plo, hi = phi;  // largest p with ppre[p] <= t
    while (hi - p > 1) {
        const uint32_t mid = (p + hi) >> 1;
        if (L.ppre[mid] <= t) p = mid; else hi = mid;
    }
    uint32_t nxt = L.ppre[p + 1], off = L.poff[p], inf = L.pinfo[p];
    while (t < t1) {
        uint32_t ent[4], pin[4];
#pragma unroll
        for (int k = 0; k < 4; k++) {
            const uint32_t tt = t + 32 * k;
            if (tt < t1) {
                if (tt >= nxt) {
                    do {
                        p++;
                        nxt = L.ppre[p + 1];
                    } while (tt >= nxt);
                    off = L.poff[p];
                    inf = L.pinfo[p];
                }
                ent[k] = B_ent[off + tt];
                pin[k] = inf;
            }
        }
#pragma unroll
        for (int k = 0; k < 4; k++)
            if (t + 32 * k < t1) fn(ent[k], pin[k]);
        t += 128;
    }
}

struct DirectOut {
    U128 sum;        // one partner: this thread's share
    RowInfo rst;     // this thread's share
    uint32_t nc = 0, nr = 0, passes = 0;
    bool failed = false;
};

// Position of the part `sdiff` of rank idx in its bitmap word: the words of 16
// ranks' counters are compared four counters at a time, byte (or half) b of
// counter word w to bit 8 b + w (8-bit counters: two ranks per word) or
// 16 b + w (16-bit counters: one).
template <bool C8>
__device__ __forceinline__ uint32_t part_bit(uint32_t idx, uint32_t sdiff) {
    if constexpr (C8) return ((idx & 1u) << 4) + (sdiff << 3) + ((idx >> 1) & 7u);
    else return (sdiff << 4) + (idx & 15u);
}

// Count of the part at bit k of bitmap word j (the counters' memory as bytes).
template <bool C8>
__device__ __forceinline__ uint32_t part_count(const unsigned char *tbl, uint32_t j, uint32_t k) {
    if constexpr (C8) return tbl[32 * j + 4 * (k & 7u) + (k >> 3)];
    else return reinterpret_cast<const uint16_t *>(tbl)[32 * j + 2 * (k & 15u) + (k >> 4)];
}

template <bool C8, bool CHECK>
__device__ __forceinline__ DirectOut direct_anchor(const TwohopArgs &a, uint32_t r, uint32_t range,
                                                unsigned char *smem, unsigned long long *warp_tot,
                                                unsigned *s_nrw, unsigned *s_ncw) {
    uint32_t *tbl = (uint32_t *)smem;
    uint32_t *bm = (uint32_t *)(smem + DT_OFF_BM), *pre = (uint32_t *)(smem + DT_OFF_PRE);
    Lists L;
    L.poff = (uint32_t *)(smem + DT_OFF_POFF);
    L.ppre = (uint32_t *)(smem + DT_OFF_PPRE);
    L.pinfo = (uint32_t *)(smem + DT_OFF_PINFO);
    L.wtot = (uint32_t *)warp_tot;
    constexpr uint32_t CELLS = C8 ? DT_CELLS8 : DT_CELLS16;
    const int tid = threadIdx.x, lane = tid & 31;
    const int l = a.l;
    const int64_t ebase = a.A_off[r];
    const int d = (int)(a.A_off[r + 1] - ebase);
    const uint32_t dp = a.dprime[r], W = (dp + 31) / 32, rsv = a.rsv_c[r];
    uint32_t *region = a.pool + a.pool_off[r];
    const uint32_t *__restrict__ B_ent = a.B_ent;
    DirectOut out;
    if (tid == 0) *s_nrw = *s_ncw = 0;
    // With at most DT_PCH positions every position has its thread: the useful
    // ones, numbered by their bit index, are staged once per window, cut to the
    // window's ranks (lists ascend by rank, so a search finds the cut).
    const bool one = d <= DT_PCH;
    uint32_t st = 0, en = 0, info = EMPTY;
    if (one && tid < d) {
        const int64_t e = ebase + tid;
        const uint32_t bit = a.A_bit[e];
        if (bit != EMPTY) {
            const uint32_t av = a.A_ent[e], y = av & VMASK;
            st = (uint32_t)(a.B_off[y] + (int64_t)a.A_pos[e] + 1);
            en = (uint32_t)a.B_off[y + 1];
            info = (av & 0x80000000u) | bit;
        }
    }
    // Positions c0 .. c0 + DT_PCH - 1 with bits in [blo, bhi), compacted.
    auto stage_batch = [&](int c0, uint32_t blo, uint32_t bhi) -> uint32_t {
        uint32_t len = 0, s0 = 0, inf = 0;
        if (c0 + tid < d) {
            const int64_t e = ebase + c0 + tid;
            const uint32_t bit = a.A_bit[e];
            if (bit >= blo && bit < bhi) {  // (EMPTY is above every bhi)
                const uint32_t av = a.A_ent[e], y = av & VMASK;
                s0 = (uint32_t)(a.B_off[y] + (int64_t)a.A_pos[e] + 1);
                len = (uint32_t)a.B_off[y + 1] - s0;
                inf = (av & 0x80000000u) | bit;
            }
        }
        uint32_t npos = 0, total = 0;
        const uint32_t slot = block_excl_scan_u32(len ? 1u : 0u, L.wtot, &npos);
        __syncthreads();
        const uint32_t ex = block_excl_scan_u32(len, L.wtot, &total);
        if (len) {
            L.ppre[slot] = ex;
            L.poff[slot] = s0 - ex;
            L.pinfo[slot] = inf;
        }
        if (tid == 0) L.ppre[npos] = total;
        __syncthreads();
        return npos;
    };
    // All entries at the bits [blo, bhi) (of the window staged last).
    auto visit = [&](uint32_t blo, uint32_t bhi, auto &&fn) {
        if (one) {
            walk_lists(L, blo, bhi, B_ent, fn);
            __syncthreads();
            return;
        }
        for (int c0 = 0; c0 < d; c0 += DT_PCH) {
            const uint32_t npos = stage_batch(c0, blo, bhi);
            if (npos) walk_lists(L, 0, npos, B_ent, fn);
            __syncthreads();
        }
    };
    for (uint32_t w0 = 0; w0 < range; w0 += CELLS) {
        const uint32_t base = r + 1 + w0, nw = range - w0 < CELLS ? range - w0 : CELLS;
        const uint32_t nbm = (nw + 15) / 16;
        auto clear = [&]() {
            for (uint32_t i = tid; i < nbm * (C8 ? 2u : 4u); i += DT_THREADS)
                reinterpret_cast<uint4 *>(tbl)[i] = make_uint4(0, 0, 0, 0);
        };
        auto count = [&](uint32_t ent, uint32_t inf) {
            const uint32_t idx = (ent & VMASK) - base;
            if (idx < nw) {
                const uint32_t sdiff = (ent ^ inf) >> 31;
                if constexpr (C8) atomicAdd(&tbl[idx >> 1], 1u << ((idx & 1u) * 16u + sdiff * 8u));
                else atomicAdd(&tbl[idx], sdiff ? 65536u : 1u);
            }
        };
        // counts
        clear();
        if (one) {
            uint32_t cut = en;
            if (w0 + CELLS < range && info != EMPTY) {  // first entry past the window
                uint32_t lo = st;
                while (lo < cut) {
                    const uint32_t mid = (lo + cut) >> 1;
                    if ((B_ent[mid] & VMASK) < base + nw) lo = mid + 1; else cut = mid;
                }
            }
            uint32_t total = 0;
            const uint32_t ex = block_excl_scan_u32(cut - st, L.wtot, &total);
            if (info != EMPTY) {
                const uint32_t slot = info & VMASK;
                L.ppre[slot] = ex;
                L.poff[slot] = st - ex;
                L.pinfo[slot] = info;
            }
            if (tid == 0) L.ppre[dp] = total;
            st = cut;
        }
        __syncthreads();
        const uint32_t nr0 = *s_nrw;
        visit(0, dp, count);
        out.passes++;
        // rows: a bit per rank and part (part_bit)
        uint32_t all = 0;     // OR (8-bit) or maximum (16-bit) of the counters: bounds the longest row
        for (uint32_t j0 = 0; j0 < nbm; j0 += DT_THREADS) {
            const uint32_t j = j0 + tid;
            uint32_t bits = 0;
            if (j < nbm) {
                if constexpr (C8) {
                    // per byte: bit 7 of (low 7 bits + 128 - l) | byte is set
                    // when the byte is at least l (l <= 8)
                    const uint32_t add = (128u - (uint32_t)l) * 0x01010101u;
#pragma unroll
                    for (int h = 0; h < 2; h++) {
                        const uint4 v = reinterpret_cast<const uint4 *>(tbl)[2 * j + h];
                        const uint32_t x[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                        for (int k = 0; k < 4; k++) {
                            const uint32_t m = (((x[k] & 0x7F7F7F7Fu) + add) | x[k]) & 0x80808080u;
                            bits |= m >> (7 - (4 * h + k));
                            all |= x[k];
                        }
                    }
                } else {
                    const uint32_t add = (32768u - (uint32_t)l) * 0x00010001u;
#pragma unroll
                    for (int h = 0; h < 4; h++) {
                        const uint4 v = reinterpret_cast<const uint4 *>(tbl)[4 * j + h];
                        const uint32_t x[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                        for (int k = 0; k < 4; k++) {
                            const uint32_t m = (((x[k] & 0x7FFF7FFFu) + add) | x[k]) & 0x80008000u;
                            bits |= m >> (15 - (4 * h + k));
                            all = __vmaxu2(all, x[k]);
                        }
                    }
                }
            }
            const uint32_t cnt = __popc(bits);
            uint32_t incl = cnt;
            if (__any_sync(FULL, bits != 0)) {
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t t = __shfl_up_sync(FULL, incl, o);
                    if (lane >= o) incl += t;
                }
                const uint32_t both = C8 ? (bits | (bits >> 8)) & 0x00FF00FFu : (bits | (bits >> 16)) & 0xFFFFu;
                const uint32_t ncw = __reduce_add_sync(FULL, (uint32_t)__popc(both));
                uint32_t at = 0;
                if (lane == 31) {
                    at = atomicAdd(s_nrw, incl);
                    atomicAdd(s_ncw, ncw);
                }
                at = __shfl_sync(FULL, at, 31) + incl - cnt;
                if (j < nbm) pre[j] = at;
                if (a.single) {
                    uint32_t b = bits;
                    while (b) {
                        const uint32_t k = __ffs(b) - 1;
                        b &= b - 1;
                        binom_add(out.sum, part_count<C8>(smem, j, k), l, &a.cnt->err);
                    }
                }
            }
            if (j < nbm) bm[j] = bits;
        }
        if constexpr (C8) all |= all >> 16;
        out.rst.longest = max(out.rst.longest, C8 ? max(all & 0xFFu, (all >> 8) & 0xFFu)
                                                  : max(all & 0xFFFFu, all >> 16));
        __syncthreads();
        const uint32_t nrw = *s_nrw - nr0;
        if (a.single || nrw == 0) {
            __syncthreads();
            continue;
        }
        if (nr0 + nrw > rsv) {
            if (tid == 0) atomicOr(&a.cnt->err, CERR_RESERVE);
            out.failed = true;
            break;
        }
        // mask words, as many at a time as the counters' memory stages
        uint32_t cw = nrw <= DT_WORDS ? DT_WORDS / nrw : 0u;
        if (cw > W) cw = W;
        const bool staged = cw > 0;
        if (!staged) cw = W;
        uint32_t hits = 0;
        for (uint32_t wa = 0; wa < W; wa += cw) {
            const uint32_t wn = W - wa < cw ? W - wa : cw;
            if (staged) {
                for (uint32_t i = tid; i < (wn * nrw + 3) / 4; i += DT_THREADS)
                    reinterpret_cast<uint4 *>(tbl)[i] = make_uint4(0, 0, 0, 0);
            } else {
                for (uint32_t i = tid; i < wn * nrw; i += DT_THREADS)
                    region[(size_t)(i / nrw) * rsv + nr0 + i % nrw] = 0;
            }
            __syncthreads();
            visit(32 * wa, 32 * (wa + wn) < dp ? 32 * (wa + wn) : dp, [&](uint32_t ent, uint32_t inf) {
                const uint32_t idx = (ent & VMASK) - base;
                if (idx >= nw) return;
                const uint32_t k = part_bit<C8>(idx, (ent ^ inf) >> 31);
                const uint32_t bw = bm[idx >> 4];
                if (!((bw >> k) & 1u)) return;
                hits++;
                const uint32_t row = pre[idx >> 4] + __popc(bw & ((1u << k) - 1u));
                const uint32_t bit = inf & VMASK, m = 1u << (bit & 31);
                if (staged) atomicOr(&tbl[((bit >> 5) - wa) * nrw + row - nr0], m);
                else atomicOr(&region[(size_t)(bit >> 5) * rsv + row], m);
            });
            if (staged) {
                if (nrw >= 64) {
                    for (uint32_t wd = 0; wd < wn; wd++)
                        for (uint32_t i = tid; i < nrw; i += DT_THREADS)
                            region[(size_t)(wa + wd) * rsv + nr0 + i] = tbl[wd * nrw + i];
                } else {
                    for (uint32_t i = tid; i < wn * nrw; i += DT_THREADS) {
                        const uint32_t wd = i / nrw;
                        region[(size_t)(wa + wd) * rsv + nr0 + (i - wd * nrw)] = tbl[i];
                    }
                }
                __syncthreads();
            }
        }
        out.rst.pops += (float)hits;
        out.passes++;
        if constexpr (CHECK) {
            // self-check: the staged words took the counters' memory, so the window
            // is counted once more; the parts with at least l positions must be
            // the rows numbered above, and every row must hold its part's count
            clear();
            __syncthreads();
            visit(0, dp, count);
            out.passes++;
            bool bad = false;
            unsigned long long words = 0;
            for (uint32_t j = tid; j < nbm; j += DT_THREADS) {
                const uint32_t bits = bm[j];
                for (uint32_t k = 0; k < 32; k++) {
                    const uint32_t x = part_count<C8>(smem, j, k);
                    const bool row = (bits >> k) & 1u;
                    bad |= row != (x >= (uint32_t)l);
                    if (!row) continue;
                    bad |= !row_matches(region + pre[j] + __popc(bits & ((1u << k) - 1u)), rsv, W, x, true);
                    words += W;
                }
            }
            if (words) atomicAdd(&a.cnt->popc_words, words);
            if (bad) atomicOr(&a.cnt->err, CERR_MASK);
            __syncthreads();
        }
    }
    __syncthreads();
    out.nr = *s_nrw;
    out.nc = *s_ncw;
    return out;
}

__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Direct counters, one CTA per anchor. (The self-check is a build of its own: its
// registers would cost the other one occupancy or spills.)
template <bool CHECK>
__global__ void __launch_bounds__(DT_THREADS, 2) k_twohop_direct(const __grid_constant__ TwohopArgs a) {
    twohop_let_next_start();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ unsigned long long warp_tot[DT_WARPS];
    __shared__ unsigned s_item, s_nrw, s_ncw, s_longest;
    __shared__ uint32_t s_rank, s_range;
    __shared__ float s_pops;
    const int tid = threadIdx.x, lane = tid & 31;
    const bool split_totals = a.tot.per_anchor || a.tot.per_graph;
    unsigned long long wedges = 0, tested = 0, leaves = 0, reads = 0, cycles = 0, anchors = 0;
    U128 sum;  // one partner: this thread's share of the sums
    // the next item is claimed, and its anchor looked up, while this one runs
    if (tid == 0) {
        s_item = a.direct_begin + atomicAdd(&a.cnt->head_direct, 1u);
        s_rank = s_item < a.direct_end ? a.order[s_item] : 0u;
    }
    for (;;) {
        __syncthreads();
        if (s_item >= a.direct_end) break;
        const uint32_t r = s_rank;
        const long long c0 = clock64();
        unsigned next = 0;
        uint32_t next_rank = 0;
        if (tid == 0) {
            next = a.direct_begin + atomicAdd(&a.cnt->head_direct, 1u);
            if (next < a.direct_end) next_rank = a.order[next];
            s_range = rank_end(a.tot.per_graph ? a.tot.graph_x0 : nullptr, a.tot.n_graphs, a.n_ranks, r) - 1 - r;
            s_pops = 0.f;
            s_longest = 0;
        }
        __syncthreads();
        DirectOut o = a.dprime[r] <= 255u
            ? direct_anchor<true, CHECK>(a, r, s_range, smem_raw, warp_tot, &s_nrw, &s_ncw)
            : direct_anchor<false, CHECK>(a, r, s_range, smem_raw, warp_tot, &s_nrw, &s_ncw);
        if (o.failed) o.nc = o.nr = 0;
        if (a.single) {
            if (sum.add(o.sum)) atomicOr(&a.cnt->err, CERR_OVERFLOW);
            if (split_totals) {
                const U128 ws = warp_sum_u128(sum, &a.cnt->err);
                if (lane == 0) add_totals(a.tot, r, ws);
                sum = U128();
            }
        } else {
            o.rst.warp_sum();
            if (lane == 0) {
                atomicAdd(&s_pops, o.rst.pops);
                atomicMax(&s_longest, o.rst.longest);
            }
            __syncthreads();
        }
        if (tid == 0) {
            a.ncand[r] = o.nc;
            a.nrow[r] = o.nr;
            RowInfo ri;
            ri.pops = s_pops;
            ri.longest = s_longest;
            a.rinfo[r] = ri;
            if (a.single) {
                tested += o.nc;
                leaves += o.nr;
            }
            wedges += a.e_use[r];
            reads += a.e_use[r] * o.passes;
            cycles += (unsigned long long)(clock64() - c0);
            anchors++;
            s_item = next;
            s_rank = next_rank;
        }
    }
    if (a.single && !split_totals) {
        const U128 ws = warp_sum_u128(sum, &a.cnt->err);
        if (lane == 0) add_totals(a.tot, 0, ws);
    }
    if (tid == 0) {
        if (wedges) atomicAdd(&a.cnt->wedges, wedges);
        if (tested) atomicAdd(&a.cnt->tested, tested);
        if (leaves) atomicAdd(&a.cnt->leaves, leaves);
        atomicAdd(&a.cnt->tw_reads, reads);
        atomicAdd(&a.cnt->tw_cyc[0], cycles);
        atomicAdd(&a.cnt->tw_anchors[0], anchors);
        const unsigned long long t = global_ns();
        atomicMax(&a.cnt->tw_fin_max, t);
        atomicMax(&a.cnt->tw_fin_min_n, ~t);
    }
    twohop_wait_previous();
}

template <bool STATS>
__global__ void __launch_bounds__(PL_THREADS, 2) k_twohop_large(const __grid_constant__ TwohopArgs a) {
    twohop_let_next_start();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    uint32_t *keys = (uint32_t *)smem_raw;
    unsigned long long *vals = (unsigned long long *)(smem_raw + PL_OFF_VALS);
    int64_t *pst = (int64_t *)(smem_raw + PL_OFF_PST);
    uint32_t *ppre = (uint32_t *)(smem_raw + PL_OFF_PPRE);
    uint32_t *pinfo = (uint32_t *)(smem_raw + PL_OFF_PINFO);
    uint32_t *stage = (uint32_t *)(smem_raw + PL_OFF_STAGE);
    __shared__ unsigned long long warp_tot[PL_WARPS];
    __shared__ unsigned long long s_total;
    __shared__ unsigned s_item, s_ncw, s_nrw, s_paper, s_ovf;
    __shared__ float s_pops;
    __shared__ uint32_t s_rank;
    __shared__ unsigned s_longest;
    __shared__ uint32_t s_bcnt[PL_MAXCLS];
    const int tid = threadIdx.x, lane = tid & 31;
    const int l = a.l;
    unsigned long long *bucket =
        a.bucket ? a.bucket + (size_t)blockIdx.x * a.bucket_slot : nullptr;
    const bool split_totals = a.tot.per_anchor || a.tot.per_graph;
    unsigned long long wedges = 0, tested = 0, leaves = 0;
    U128 sum;  // one partner: this thread's share of the anchor's sum
    RowInfo rst;

    // Candidate filter over the table, window-local row indices in vals.
    auto extract = [&](uint32_t hs) {
        for (uint32_t base = 0; base < hs; base += PL_THREADS) {
            uint32_t i = base + tid;
            bool same = false, diff = false, pap = false;
            unsigned long long v = 0;
            if (i < hs && keys[i] != EMPTY) {
                v = vals[i];
                pap = STATS && (v & M21) >= (unsigned long long)l;
                same = keep_same(v, l);
                diff = keep_diff(v, l);
            }
            const uint32_t bs = __ballot_sync(FULL, same), bd = __ballot_sync(FULL, diff);
            const uint32_t pb = __ballot_sync(FULL, pap);
            uint32_t wbase = 0;
            if (lane == 0 && (bs | bd)) {
                wbase = atomicAdd(&s_nrw, (unsigned)(__popc(bs) + __popc(bd)));
                atomicAdd(&s_ncw, (unsigned)__popc(bs | bd));
            }
            if (lane == 0 && pb) atomicAdd(&s_paper, (unsigned)__popc(pb));
            wbase = __shfl_sync(FULL, wbase, 0);
            const uint32_t lt = (1u << lane) - 1u;
            if (same || diff) vals[i] = cand_value(v, wbase + __popc(bs & lt) + __popc(bd & lt));
            if (a.single) {
                if (same) binom_add(sum, use_count(v) - diff_count(v), l, &a.cnt->err);
                if (diff) binom_add(sum, diff_count(v), l, &a.cnt->err);
            } else {
                if (same) rst.add(use_count(v) - diff_count(v));
                if (diff) rst.add(diff_count(v));
            }
        }
    };
    auto set_bits = [&](uint32_t hs, uint32_t *bb, uint32_t bstride, uint32_t w, uint32_t sdiff,
                        uint32_t bit) {
        int sl = tab_find(keys, hs, w);
        if (sl < 0) return;
        unsigned long long v = vals[sl];
        if (!(v & CAND)) return;
        const uint32_t row = row_index(v, sdiff, l);
        if (row != EMPTY) atomicOr(&bb[(size_t)(bit >> 5) * bstride + row], 1u << (bit & 31));
    };

    // the next item is claimed, and its anchor looked up, while this one runs
    if (tid == 0) {
        s_item = a.large_begin + atomicAdd(&a.cnt->head_large, 1u);
        s_rank = s_item < a.large_end ? a.order[s_item] : 0u;
    }
    for (;;) {
        __syncthreads();
        const unsigned item = s_item;
        if (item >= a.large_end) break;
        const uint32_t r = s_rank;
        __syncthreads();
        unsigned next = 0;
        uint32_t next_rank = 0;
        if (tid == 0) {
            next = a.large_begin + atomicAdd(&a.cnt->head_large, 1u);
            if (next < a.large_end) next_rank = a.order[next];
        }
        const int64_t ebase = a.A_off[r];
        const int d = (int)(a.A_off[r + 1] - ebase);
        const uint32_t W = (a.dprime[r] + 31) / 32;
        const uint32_t rsv = a.rsv_c[r];
        uint32_t *region = a.pool + a.pool_off[r];
        const unsigned long long e_vis = STATS ? a.e_all[r] : a.e_use[r];
        const unsigned long long e_use = a.e_use[r];
        const long long c0 = clock64();
        unsigned long long reads = 0;
        int path = 0;
        uint32_t nc = 0, nr = 0, npaper = 0;
        bool failed = false;
        rst = RowInfo();
        if (tid == 0) {
            s_pops = 0.f;
            s_longest = 0;
        }

        // Window bookkeeping shared by both strategies: after the table of
        // one window holds its counts, keep candidates and write their bits.
        // Returns false when the reservation would overflow.
        auto finish_window = [&](uint32_t hs, auto &&pass2) -> bool {
            extract(hs);
            __syncthreads();
            const uint32_t ncw = s_ncw, nrw = s_nrw;
            npaper += s_paper;
            if (nrw > 0 && !a.single) {
                if (nr + nrw > rsv) {
                    if (tid == 0) atomicOr(&a.cnt->err, CERR_RESERVE);
                    __syncthreads();
                    return false;
                }
                const bool staged = (unsigned long long)W * nrw <= (unsigned long long)PL_STAGE_WORDS;
                uint32_t *bb = staged ? stage : region + nr;
                const uint32_t bstride = staged ? nrw : rsv;
                for (uint32_t i = tid; i < W * nrw; i += PL_THREADS) {
                    uint32_t wd = i / nrw, c = i % nrw;
                    bb[(size_t)wd * bstride + c] = 0;
                }
                __syncthreads();
                pass2(bb, bstride);
                __syncthreads();
                if (a.check) {
                    bool bad = false;
                    unsigned long long words = 0;
                    for (uint32_t i = tid; i < hs; i += PL_THREADS) {
                        if (keys[i] == EMPTY) continue;
                        const unsigned long long v = vals[i];
                        if ((v & CAND) && !rows_match(bb, bstride, W, v, l, !staged, words)) bad = true;
                    }
                    if (words) atomicAdd(&a.cnt->popc_words, words);
                    if (bad) atomicOr(&a.cnt->err, CERR_MASK);
                    __syncthreads();
                }
                if (staged) {
                    for (uint32_t i = tid; i < W * nrw; i += PL_THREADS) {
                        uint32_t wd = i / nrw, c = i % nrw;
                        region[(size_t)wd * rsv + nr + c] = stage[i];
                    }
                }
            }
            nc += ncw;
            nr += nrw;
            __syncthreads();
            return true;
        };
        auto clear_table = [&](uint32_t hs) {
            for (uint32_t i = tid; i < hs; i += PL_THREADS) {
                keys[i] = EMPTY;
                vals[i] = 0;
            }
            if (tid == 0) {
                s_ncw = 0;
                s_nrw = 0;
                s_paper = 0;
                s_ovf = 0;
            }
            __syncthreads();
        };

        const int lgb = bucket_lg(e_vis);
        bool bucketed = false;
        if (e_vis <= (unsigned long long)a.wcap) {
            // one window
            uint32_t hs = (uint32_t)((2 * e_vis + 31) & ~31ull);
            hs = hs < 64 ? 64 : (hs > PL_HS ? PL_HS : hs);
            hs = cap_slots(hs, a);
            clear_table(hs);
            reads = e_vis + e_use;
            visit_block(ebase, d, !STATS, 0, 0, a, pst, ppre, pinfo, warp_tot, &s_total,
                        [&](uint32_t w, uint32_t sdiff, uint32_t bit) {
                            if (!tab_insert(keys, vals, hs, w, pass1_add(sdiff, bit))) s_ovf = 1;
                        });
            if (s_ovf) {
                failed = true;
                if (tid == 0) atomicOr(&a.cnt->err, CERR_HASH);
            } else {
                failed = !finish_window(hs, [&](uint32_t *bb, uint32_t bstride) {
                    visit_block(ebase, d, true, 0, 0, a, pst, ppre, pinfo, warp_tot, &s_total,
                                [&](uint32_t w, uint32_t sdiff, uint32_t bit) {
                                    set_bits(hs, bb, bstride, w, sdiff, bit);
                                });
                });
            }
        } else if (bucket && lgb <= 10 &&
                   (bucket_cap(e_vis, lgb) << lgb) <= a.bucket_slot) {
            // partition the wedges once into 2^lgb hash classes, then one
            // window per class from its bucket
            const uint32_t ncls = 1u << lgb;
            const uint32_t cap = (uint32_t)bucket_cap(e_vis, lgb);
            for (uint32_t i = tid; i < ncls; i += PL_THREADS) s_bcnt[i] = 0;
            if (tid == 0) s_ovf = 0;
            __syncthreads();
            visit_block(ebase, d, !STATS, 0, 0, a, pst, ppre, pinfo, warp_tot, &s_total,
                        [&](uint32_t w, uint32_t sdiff, uint32_t bit) {
                            uint32_t c = class_of(w, lgb);
                            uint32_t pos = atomicAdd(&s_bcnt[c], 1u);
                            if (pos < cap) bucket[(size_t)c * cap + pos] = bucket_entry(w, sdiff, bit);
                            else s_ovf = 1;
                        });
            reads = e_vis;
            path = 1;
            __syncthreads();
            // A partner sharing many of the anchor's positions fills its class
            // beyond the capacity. The class sizes are exact all the same, so
            // the wedges are then scattered once more, classes back to back.
            const bool packed = s_ovf != 0;
            if (packed) {
                uint32_t *cursor = keys;  // the table is free until the windows
                const uint32_t c2 = 2 * tid;
                const uint32_t n0 = c2 < ncls ? s_bcnt[c2] : 0u;
                const uint32_t n1 = c2 + 1 < ncls ? s_bcnt[c2 + 1] : 0u;
                const unsigned long long ex = block_excl_scan_u64(n0 + n1, warp_tot, &s_total);
                if (c2 < ncls) cursor[c2] = (uint32_t)ex;
                if (c2 + 1 < ncls) cursor[c2 + 1] = (uint32_t)ex + n0;
                __syncthreads();
                visit_block(ebase, d, !STATS, 0, 0, a, pst, ppre, pinfo, warp_tot, &s_total,
                            [&](uint32_t w, uint32_t sdiff, uint32_t bit) {
                                uint32_t pos = atomicAdd(&cursor[class_of(w, lgb)], 1u);
                                bucket[pos] = bucket_entry(w, sdiff, bit);
                            });
                reads += e_vis;
                path = 3;
                __syncthreads();
            }
            bucketed = true;
            size_t base = 0;
            for (uint32_t c = 0; c < ncls && !failed; c++) {
                const uint32_t n = s_bcnt[c];
                const unsigned long long *bk = bucket + (packed ? base : (size_t)c * cap);
                base += n;
                if (n == 0) continue;
                // one window for the class; when its distinct partners overflow
                // the table, 2^lg2 windows over its sub-classes
                const uint32_t nc0 = nc, nr0 = nr, np0 = npaper;
                const U128 sum0 = sum;
                const RowInfo rst0 = rst;
                for (int lg2 = 0; !failed; lg2++) {
                    if (lg2 > 8) {
                        if (tid == 0) atomicOr(&a.cnt->err, CERR_HASH);
                        failed = true;
                        break;
                    }
                    const uint32_t per = (n + (1u << lg2) - 1) >> lg2;
                    uint32_t hs = (uint32_t)((2ull * per + 31) & ~31ull);
                    hs = hs < 64 ? 64 : (hs > PL_HS ? PL_HS : hs);
                    hs = cap_slots(hs, a);
                    nc = nc0;
                    nr = nr0;
                    npaper = np0;
                    sum = sum0;
                    rst = rst0;
                    bool over = false;
                    for (uint32_t sub = 0; sub < (1u << lg2) && !failed; sub++) {
                        __syncthreads();
                        clear_table(hs);
                        for (uint32_t i = tid; i < n; i += PL_THREADS) {
                            unsigned long long e = bk[i];
                            const uint32_t w = (uint32_t)e & VMASK;
                            if (lg2 && subclass_of(w, lgb, lg2) != sub) continue;
                            uint32_t bi = (uint32_t)(e >> 32);
                            uint32_t bit = bi == (uint32_t)BE_NOBIT ? EMPTY : bi;
                            if (!tab_insert(keys, vals, hs, w, pass1_add((uint32_t)(e >> 31) & 1u, bit)))
                                s_ovf = 1;
                        }
                        __syncthreads();
                        if (s_ovf) {
                            over = true;
                            break;
                        }
                        failed = !finish_window(hs, [&](uint32_t *bb, uint32_t bstride) {
                            for (uint32_t i = tid; i < n; i += PL_THREADS) {
                                unsigned long long e = bk[i];
                                uint32_t bi = (uint32_t)(e >> 32);
                                if (bi == (uint32_t)BE_NOBIT) continue;
                                const uint32_t w = (uint32_t)e & VMASK;
                                if (lg2 && subclass_of(w, lgb, lg2) != sub) continue;
                                set_bits(hs, bb, bstride, w, (uint32_t)(e >> 31) & 1u, bi);
                            }
                        });
                    }
                    if (!over) break;
                    if (lg2 == 0 && tid == 0) atomicAdd(&a.cnt->tw_split, 1ull);
                }
            }
        }
        if (!bucketed && !failed && e_vis > (unsigned long long)a.wcap) {
            // re-read windows: every pass over the 2-hop keeps one hash class
            const U128 sum0 = sum;
            int lg_nw = 0;
            while (((unsigned long long)a.wcap << lg_nw) < e_vis) lg_nw++;
            path = 2;
            for (int attempt = 0; attempt < 8 && !failed; attempt++) {
                const uint32_t nw = 1u << lg_nw;
                reads += (unsigned long long)nw * (e_vis + e_use);
                const unsigned long long per = (e_vis + nw - 1) >> lg_nw;
                uint32_t hs = (uint32_t)((2 * per + 31) & ~31ull);
                hs = hs < 64 ? 64 : (hs > PL_HS ? PL_HS : hs);
                hs = cap_slots(hs, a);
                nc = nr = 0;
                npaper = 0;
                sum = sum0;
                rst = RowInfo();
                bool restart = false;
                for (uint32_t cls = 0; cls < nw && !failed; cls++) {
                    clear_table(hs);
                    visit_block(ebase, d, !STATS, lg_nw, cls, a, pst, ppre, pinfo, warp_tot,
                                &s_total, [&](uint32_t w, uint32_t sdiff, uint32_t bit) {
                                    if (!tab_insert(keys, vals, hs, w, pass1_add(sdiff, bit)))
                                        s_ovf = 1;
                                });
                    if (s_ovf) {
                        restart = true;
                        break;
                    }
                    failed = !finish_window(hs, [&](uint32_t *bb, uint32_t bstride) {
                        visit_block(ebase, d, true, lg_nw, cls, a, pst, ppre, pinfo, warp_tot,
                                    &s_total, [&](uint32_t w, uint32_t sdiff, uint32_t bit) {
                                        set_bits(hs, bb, bstride, w, sdiff, bit);
                                    });
                    });
                }
                if (!restart) break;
                lg_nw++;
                if (attempt == 7) {
                    if (tid == 0) atomicOr(&a.cnt->err, CERR_HASH);
                    failed = true;
                }
                __syncthreads();
            }
        }
        if (failed) nc = nr = 0;
        if (!a.single) {
            rst.warp_sum();
            if (lane == 0) {
                atomicAdd(&s_pops, rst.pops);
                atomicMax(&s_longest, rst.longest);
            }
            __syncthreads();
        }
        if (a.single && split_totals) {
            const U128 ws = warp_sum_u128(sum, &a.cnt->err);
            if (lane == 0) add_totals(a.tot, r, ws);
            sum = U128();
        }
        if (tid == 0) {
            a.ncand[r] = nc;
            a.nrow[r] = nr;
            RowInfo ri;
            ri.pops = s_pops;
            ri.longest = s_longest;
            a.rinfo[r] = ri;
            if (a.single) {
                tested += nc;
                leaves += nr;
            }
            if (STATS) a.npaper[r] = npaper;
            wedges += e_vis;
            atomicAdd(&a.cnt->tw_reads, reads);
            atomicAdd(&a.cnt->tw_cyc[path], (unsigned long long)(clock64() - c0));
            atomicAdd(&a.cnt->tw_anchors[path], 1ull);
            s_item = next;
            s_rank = next_rank;
        }
    }
    if (a.single && !split_totals) {
        const U128 ws = warp_sum_u128(sum, &a.cnt->err);
        if (lane == 0) add_totals(a.tot, 0, ws);
    }
    if (tid == 0) {
        if (wedges) atomicAdd(&a.cnt->wedges, wedges);
        if (tested) atomicAdd(&a.cnt->tested, tested);
        if (leaves) atomicAdd(&a.cnt->leaves, leaves);
        if (a.direct_begin == a.direct_end) {  // (else the direct kernel's are taken)
            const unsigned long long t = global_ns();
            atomicMax(&a.cnt->tw_fin_max, t);
            atomicMax(&a.cnt->tw_fin_min_n, ~t);
        }
    }
    twohop_wait_previous();
}

// ------------------------------------------------------------------ groups

// Pool words of the ordered anchors: gw[i] = words of order[i].
__global__ void k_gather_words(const uint32_t *order, const uint32_t *dprime, const uint32_t *rsv_c,
                               int64_t n, int64_t *gw) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i <= n;
         i += (int64_t)gridDim.x * blockDim.x)
        gw[i] = i < n ? (int64_t)((dprime[order[i]] + 31) / 32) * rsv_c[order[i]] : 0;
}

// Pool offsets of one group of sorted anchors [a, b): offset from cum[a].
__global__ void k_group_offsets(const uint32_t *order, const int64_t *cum, int64_t a, int64_t b,
                                int64_t *pool_off) {
    for (int64_t i = a + blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < b;
         i += (int64_t)gridDim.x * blockDim.x)
        pool_off[order[i]] = cum[i] - cum[a];
}

#include "tuples.cuh"

}  // namespace

// ------------------------------------------------------------------ host side

namespace {

// Relative cost of one prefix node of the column walk (per row word per lane)
// against one mask word of the row enumeration; measured on GB300.
constexpr unsigned long long kPosNodeCost = 3;
// Default tuple work items per half of a resident CTA of a full launch.
constexpr unsigned long long kSplitPerWarp = 4;
// Two-partner anchors with at least this many mask words and candidates take
// the tensor-core pair step. A 128-position step is mostly empty for one word,
// but a pair of rows still costs less there than in the tuple kernel: (4,3) of
// the 500k-edge graph 5.4 + 0.8 ms (row pairs of one-word anchors + tensor
// cores) with 2 words, 0.4 + 2.2 ms with 1; (3,3) of the 2M-edge graph
// 2.0 + 3.1 and 0.7 + 3.6 ms.
constexpr uint32_t kTcMinWords = 1;
constexpr uint32_t kTcMinCandidates = 128;

// Largest x with binom(x, l) computable in 64 bits by the multiplicative
// formula: every partial product binom(x-l+i, i) * i must stay below 2^64.
unsigned long long binom64_limit(int l) {
    auto fits = [l](unsigned long long x) {
        unsigned __int128 r = 1;
        for (int i = 1; i <= l; i++) {
            unsigned __int128 prod = r * (unsigned __int128)(x - l + i);
            if (prod >> 64) return false;
            r = prod / i;
        }
        return true;
    };
    unsigned long long lo = (unsigned long long)l, hi = 1ull << 40;
    while (lo < hi) {
        unsigned long long mid = lo + (hi - lo + 1) / 2;
        if (fits(mid)) lo = mid; else hi = mid - 1;
    }
    return lo;
}

template <int R>
void set_tuple_attr() {
    SBC_CUDA(cudaFuncSetAttribute(k_tuples<R>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)TU_SMEM));
}

// Opt every large-shared-memory kernel in, and load the binomial limits,
// once per device.
void ensure_kernel_attrs() {
    static std::mutex mu;
    static bool done[64] = {};
    std::lock_guard<std::mutex> lock(mu);
    int dev = 0;
    SBC_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) fail(SBC_E_UNSUPPORTED, "device ordinal %d out of range", dev);
    if (done[dev]) return;
    // Counts allocate and free their buffers (plans, candidate pools, the
    // tensor-core Z arena) on the stream from the device's default memory
    // pool; let the pool keep up to 4 GiB of freed memory mapped between
    // counts instead of returning it at every synchronisation.
    {
        cudaMemPool_t pool;
        if (cudaDeviceGetDefaultMemPool(&pool, dev) == cudaSuccess) {
            uint64_t keep = 4ull << 30, cur = 0;
            if (cudaMemPoolGetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &cur) == cudaSuccess &&
                cur < keep)
                SBC_CUDA(cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep));
        }
        cudaGetLastError();
    }
    unsigned long long lim[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
    for (int i = 2; i <= 8; i++) lim[i] = binom64_limit(i);
    SBC_CUDA(cudaMemcpyToSymbol(c_binom64_max, lim, sizeof(lim)));
    SBC_CUDA(cudaFuncSetAttribute(k_twohop_small<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PS_SMEM));
    SBC_CUDA(cudaFuncSetAttribute(k_twohop_small<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PS_SMEM));
    SBC_CUDA(cudaFuncSetAttribute(k_twohop_direct<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)DT_SMEM));
    SBC_CUDA(cudaFuncSetAttribute(k_twohop_direct<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)DT_SMEM));
    SBC_CUDA(cudaFuncSetAttribute(k_twohop_large<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PL_SMEM));
    SBC_CUDA(cudaFuncSetAttribute(k_twohop_large<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PL_SMEM));
    tc_ensure_attrs();
    set_tuple_attr<2>();
    set_tuple_attr<3>();
    set_tuple_attr<4>();
    set_tuple_attr<5>();
    set_tuple_attr<6>();
    set_tuple_attr<7>();
    done[dev] = true;
}

template <int R>
void launch_tuples(int grid, cudaStream_t s, const TupleArgs &a) {
    k_tuples<R><<<grid, TU_THREADS, TU_SMEM, s>>>(a);
    SBC_LAUNCHED();
}

int blocks_per_sm(const void *fn, int threads, size_t smem) {
    int n = 0;
    SBC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fn, threads, smem));
    return n < 1 ? 1 : n;
}


}  // namespace

struct EventTimer {
    cudaEvent_t e[5] = {nullptr, nullptr, nullptr, nullptr, nullptr};
    bool on;
    explicit EventTimer(bool enable) : on(enable) {
        if (on)
            for (auto &x : e) SBC_CUDA(cudaEventCreate(&x));
    }
    void mark(int i, cudaStream_t s) {
        if (on) SBC_CUDA(cudaEventRecord(e[i], s));
    }
    float ms(int a, int b) {
        float t = 0;
        if (on) SBC_CUDA(cudaEventElapsedTime(&t, e[a], e[b]));
        return t;
    }
    ~EventTimer() {
        for (auto &x : e)
            if (x) cudaEventDestroy(x);
    }
};

struct CountRun {
    const Orient *o = nullptr;
    int64_t nnz = 0, nX = 0;
    CountSpec spec;
    int R = 0;
    cudaStream_t s = nullptr;
    DevBuf<Counters> cnt;
    DevBuf<unsigned char> ws;       // per-anchor and per-entry arrays, one allocation
    uint32_t *A_bit = nullptr, *dprime = nullptr, *rsv_c = nullptr, *order = nullptr, *ncand = nullptr,
             *nrow = nullptr, *npaper = nullptr;
    unsigned long long *e_use = nullptr, *e_all = nullptr;
    int64_t *pool_off = nullptr;
    RowInfo *rinfo = nullptr;
    DevBuf<uint32_t> pool, claims, scratch, warp_list;
    DevBuf<unsigned long long> bucket, per;
    DevBuf<int64_t> cum_dev;
    DevBuf<Item> items;
    DevBuf<TcInput> tc_in;
    DevBuf<unsigned char> zbuf;     // Z arena of the tensor-core pair step
    std::vector<TcPlan> tc_plans;   // per anchor group
    TwohopArgs ta;
    TupleArgs tu;
    int gd = 0, ga = 0, gs = 0, gt = 0;
    int64_t n_items = 0;
    Counters hc;
    CountResult res;

    // Launches that execute a planned count (no host synchronisation, no
    // allocation): usable under stream capture. Valid when the plan has at
    // most one anchor group.
    void launch_count() {
        SBC_CUDA(cudaMemsetAsync(&cnt.ptr->run_begin, 0,
                                 sizeof(Counters) - offsetof(Counters, run_begin), s));
        if (per.ptr) SBC_CUDA(cudaMemsetAsync(per.ptr, 0, per.bytes(), s));
        if (spec.per_graph) SBC_CUDA(cudaMemsetAsync(spec.per_graph, 0, 16 * (size_t)spec.n_graphs, s));
        if (groups.empty()) return;
        zero_pool(0);
        launch_twohop((unsigned)groups[0].first, (unsigned)groups[0].second);
        if (claims.ptr) SBC_CUDA(cudaMemsetAsync(claims.ptr, 0, claims.bytes(), s));
        if (gt > 0) launch_tuple_kernel();
        launch_tc(0);
    }

    // Tensor-core pair step of group `grp` (expansion and pair kernels of each
    // of its chunks).
    void launch_tc(size_t grp) {
        if (grp >= tc_plans.size() || tc_plans[grp].anchors == 0) return;
        TcArgs ta2;
        ta2.pool = pool.ptr;
        ta2.l = spec.l;
        ta2.total = cnt.ptr->total;
        ta2.per_anchor = per.ptr;
        ta2.per_graph = spec.per_graph;
        ta2.graph_x0 = spec.graph_x0;
        ta2.n_graphs = spec.n_graphs;
        ta2.err = &cnt.ptr->err;
        ta2.big64 = binom64_limit(spec.l);
        tc_launch(tc_plans[grp], ta2, zbuf.ptr, s);
    }

    // Bytes of Z one tensor-core chunk may take.
    int64_t tc_budget_bytes() const {
        size_t fr = 0, tot = 0;
        SBC_CUDA(cudaMemGetInfo(&fr, &tot));
        int64_t b = (int64_t)(fr / 8);
        return std::max<int64_t>(256ll << 20, std::min<int64_t>(b, kTcArenaMax));
    }

    // Events around the 2-hop and tuple launches of each group (pairs).
    std::vector<cudaEvent_t> ev_twohop, ev_tuples;
    cudaEvent_t new_event(std::vector<cudaEvent_t> &v) {
        cudaEvent_t e = nullptr;
        SBC_CUDA(cudaEventCreate(&e));
        v.push_back(e);
        return e;
    }
    void drop_events() {
        for (cudaEvent_t e : ev_twohop) cudaEventDestroy(e);
        for (cudaEvent_t e : ev_tuples) cudaEventDestroy(e);
        for (cudaEvent_t e : ev_tc) cudaEventDestroy(e);
        ev_twohop.clear();
        ev_tuples.clear();
        ev_tc.clear();
    }
    static float pairs_ms(const std::vector<cudaEvent_t> &v) {
        float sum = 0;
        for (size_t i = 0; i + 1 < v.size(); i += 2) {
            float t = 0;
            SBC_CUDA(cudaEventElapsedTime(&t, v[i], v[i + 1]));
            sum += t;
        }
        return sum;
    }
    ~CountRun() { drop_events(); }

    // Device words the candidate pool may take at once.
    int64_t pool_budget_words() const {
        if (const char *e = getenv("SBC_POOL_BUDGET_KB")) {  // tuning / testing override
            long long v = atoll(e);
            if (v > 0) return (int64_t)v * 256;
        }
        // the fixed scratch of the no-allocation entry point frees only its
        // top allocation: one group there
        if (thread_arena_active()) return INT64_MAX / 8;
        size_t fr = 0, tot = 0;
        SBC_CUDA(cudaMemGetInfo(&fr, &tot));
        return (int64_t)(fr / 4 / 4);
    }

    // The warp tier of the 2-hop step builds its rows with atomicOr into words
    // that are zero on entry; the CTA tier clears or writes every word it uses.
    void zero_pool(size_t grp) {
        int64_t from = words_big, words = words_small;
        if (!cum.empty()) {
            const int64_t a = groups[grp].first, b = groups[grp].second;
            const int64_t f = std::min(std::max<int64_t>(a, hc.n_big), b);
            from = cum[f] - cum[a];
            words = cum[b] - cum[f];
        }
        if (words > 0) SBC_CUDA(cudaMemsetAsync(pool.ptr + from, 0, (size_t)words * 4, s));
    }

    void launch_twohop(unsigned a, unsigned b) {
        ta.direct_begin = a;
        ta.direct_end = b < hc.n_direct ? b : hc.n_direct;
        ta.large_begin = a > hc.n_direct ? a : hc.n_direct;
        ta.large_end = b < hc.n_big ? b : hc.n_big;
        ta.small_begin = a > hc.n_big ? a : hc.n_big;
        ta.small_end = b;
        // The kernels fill disjoint anchors' rows, so each may start where the one
        // before it leaves room (every CTA of which runs by then) and ends after it:
        // the few hub anchors left to the hash kernel, first, no longer run alone
        // (2-hop of the (2,2) count of the 2M-edge graph 7.4 -> 5.6 ms).
        bool after = false;  // a 2-hop kernel is the last work on the stream
        if (ga > 0 && ta.large_end > ta.large_begin)
            launch_overlapped(spec.paper ? k_twohop_large<true> : k_twohop_large<false>, ga,
                              ta.large_end - ta.large_begin, PL_THREADS, PL_SMEM, after);
        if (ta.direct_end > ta.direct_begin)
            launch_overlapped(spec.check ? k_twohop_direct<true> : k_twohop_direct<false>, gd, ta.direct_end - ta.direct_begin, DT_THREADS, DT_SMEM, after);
        if (gs > 0 && ta.small_end > ta.small_begin)
            launch_overlapped(spec.paper ? k_twohop_small<true> : k_twohop_small<false>, gs,
                              (ta.small_end - ta.small_begin + PS_WARPS - 1) / PS_WARPS, PS_THREADS, PS_SMEM,
                              after);
    }

    void launch_overlapped(void (*k)(TwohopArgs), int grid, unsigned need, int threads, size_t smem, bool &after) {
        cudaLaunchAttribute at = {};
        at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at.val.programmaticStreamSerializationAllowed = 1;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)grid > need ? need : (unsigned)grid);
        cfg.blockDim = dim3((unsigned)threads);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = s;
        cfg.attrs = &at;
        cfg.numAttrs = after ? 1 : 0;
        SBC_CUDA(cudaLaunchKernelEx(&cfg, k, ta));
        g_launches++;
        after = true;
    }

    void launch_tuple_kernel() {
        switch (R) {
            case 2: launch_tuples<2>(gt, s, tu); break;
            case 3: launch_tuples<3>(gt, s, tu); break;
            case 4: launch_tuples<4>(gt, s, tu); break;
            case 5: launch_tuples<5>(gt, s, tu); break;
            case 6: launch_tuples<6>(gt, s, tu); break;
            default: launch_tuples<7>(gt, s, tu); break;
        }
        g_launches++;
    }

    std::vector<std::pair<int64_t, int64_t>> groups;  // ranges of the sorted anchors
    bool several = false;      // more than one (kept while a new plan is made, which may fail)
    int64_t words_big = 0, words_small = 0;  // pool words of the two 2-hop tiers
    std::vector<int64_t> cum;  // several groups: pool words before each ordered anchor
    float tw_tail_ms = 0;      // largest finish spread of the CTA-wide 2-hop kernel's CTAs

    // Finish spread of the CTA-wide 2-hop launch of the last group (counters in hc).
    float group_tail_ms() const {
        return hc.tw_fin_max ? (float)((double)(hc.tw_fin_max - ~hc.tw_fin_min_n) * 1e-6) : 0.f;
    }
    float ms_twohop = 0, ms_tuples = 0, ms_tc = 0;
    std::vector<cudaEvent_t> ev_tc;

    // Tensor-core plan of group `grp`.
    void plan_tc(size_t grp, const std::vector<TcInput> &in) {
        TcPlan plan = tc_plan(in, spec.l, tc_budget_bytes());
        tc_upload(plan, s);
        const size_t need = (size_t)plan.max_blocks * (size_t)kTcBlockBytes;
        if (need > zbuf.bytes()) zbuf.alloc(need, s);
        tc_anchors += (uint64_t)plan.anchors;
        tc_tiles += (uint64_t)plan.tiles;
        tc_kblocks += plan.kblocks;
        tc_plans[grp] = std::move(plan);
    }

    void run_tc_timed(size_t grp, bool timing) {
        if (grp >= tc_plans.size() || tc_plans[grp].anchors == 0) return;
        cudaEvent_t t4 = timing ? new_event(ev_tc) : nullptr;
        cudaEvent_t t5 = timing ? new_event(ev_tc) : nullptr;
        if (t4) SBC_CUDA(cudaEventRecord(t4, s));
        NvtxRange nr("sbc/tc_pairs");
        launch_tc(grp);
        if (t5) SBC_CUDA(cudaEventRecord(t5, s));
    }
    uint64_t tc_anchors = 0, tc_tiles = 0, tc_kblocks = 0;

    // Plan (with host reads of sizes) and execute once. Anchors are taken in
    // heavy-first order in groups whose rows fit the pool budget; each group runs
    // its 2-hop kernels, item planning, tuple kernel and tensor-core step.
    void plan_and_run(EventTimer *tm) {
        NvtxRange nr("sbc/count");
        FreeOnStream frees(s);  // (a plan made again drops the one before it)
        const bool timing = tm != nullptr;
        const int B = 256;
        groups.clear();
        drop_events();
        tc_anchors = tc_tiles = tc_kblocks = 0;
        ta.direct_begin = ta.direct_end = ta.large_begin = ta.large_end = ta.small_begin = ta.small_end = 0;
        gt = 0;
        const int l = spec.l;
        R = spec.k - 1;
        // one allocation for the arrays, its head zeroed: counters' histogram
        // and cursors, ncand, nrow, npaper
        cnt.alloc(1, s);
        SBC_CUDA(cudaMemsetAsync(cnt.ptr, 0, sizeof(Counters), s));
        size_t at = 0;
        auto carve = [&](size_t bytes) {
            const size_t p = at;
            at += (bytes + 255) & ~(size_t)255;
            return p;
        };
        const size_t N = (size_t)nX;
        const size_t o_words = carve(16), o_hist = carve(1024), o_cursor = carve(1024), o_ncand = carve(4 * N),
                     o_nrow = carve(4 * N), o_npaper = carve(spec.paper ? 4 * N : 0), zeroed = at,
                     o_bit = carve(4 * (size_t)nnz), o_dprime = carve(4 * N), o_rsv = carve(4 * N),
                     o_order = carve(4 * N), o_use = carve(8 * N), o_all = carve(spec.paper ? 8 * N : 0),
                     o_off = carve(8 * N), o_info = carve(sizeof(RowInfo) * N), o_key = carve(N);
        ws.alloc(at, s);
        unsigned char *w = ws.ptr;
        unsigned long long *word_cursor = (unsigned long long *)(w + o_words);
        uint32_t *hist = (uint32_t *)(w + o_hist), *cursor = (uint32_t *)(w + o_cursor);
        ncand = (uint32_t *)(w + o_ncand);
        nrow = (uint32_t *)(w + o_nrow);
        npaper = spec.paper ? (uint32_t *)(w + o_npaper) : nullptr;
        A_bit = (uint32_t *)(w + o_bit);
        dprime = (uint32_t *)(w + o_dprime);
        rsv_c = (uint32_t *)(w + o_rsv);
        order = (uint32_t *)(w + o_order);
        e_use = (unsigned long long *)(w + o_use);
        e_all = spec.paper ? (unsigned long long *)(w + o_all) : nullptr;
        pool_off = (int64_t *)(w + o_off);
        rinfo = (RowInfo *)(w + o_info);
        uint8_t *key = w + o_key;
        SBC_CUDA(cudaMemsetAsync(w, 0, zeroed, s));
        PlanArgs pa;
        pa.A_off = o->A_off.ptr;
        pa.A_ent = o->A_ent.ptr;
        pa.A_pos = o->A_pos.ptr;
        pa.B_off = o->B_off.ptr;
        pa.nX = nX;
        pa.R = R;
        pa.l = l;
        pa.shard = spec.shard;
        pa.nshard = spec.nshard;
        pa.stats = spec.paper ? 1 : 0;
        pa.small_e = spec.small_e > 0 ? spec.small_e : SMALL_E_MAX;
        pa.direct = hash_slots_cap() == 0 && twohop_window_wedges() == (uint32_t)PL_WCAP;
        pa.graph_x0 = spec.per_graph ? spec.graph_x0 : nullptr;
        pa.n_graphs = spec.n_graphs;
        pa.A_bit = A_bit;
        pa.dprime = dprime;
        pa.rsv_c = rsv_c;
        pa.e_use = e_use;
        pa.e_all = e_all;
        pa.key = key;
        pa.hist = hist;
        pa.cnt = cnt.ptr;
        // Full chunks, but on a side with rows for the CTA enough chunks to give few
        // anchors a CTA each (plan of 60 anchors of 50,000 entries: 4.2 ms on two
        // CTAs, 0.2 on sixty)
        const int64_t full = (nX + PLAN_ROWS - 1) / PLAN_ROWS;
        pa.chunks = o->max_deg_x > PLAN_WARP ? std::max(full, std::min<int64_t>(nX, 4 * sm_count())) : full;
        k_plan<<<(int)std::min<int64_t>(pa.chunks, 152 * 8), PLAN_THREADS, 0, s>>>(pa);
        SBC_LAUNCHED();
        k_order<<<grid_for(nX, 256, 152 * 8), 256, 0, s>>>(key, nX, hist, dprime, rsv_c, cursor, word_cursor,
                                                           cnt.ptr, order, pool_off);
        SBC_LAUNCHED();
        g_launches += 2;
        SBC_CUDA(cudaMemcpyAsync(&hc, cnt.ptr, sizeof(Counters), cudaMemcpyDeviceToHost, s));
        SBC_CUDA(cudaStreamSynchronize(s));
        const int64_t n_act = hc.n_active;
        words_big = (int64_t)hc.words_big;
        words_small = (int64_t)hc.words_small;
        cum.clear();
        const int64_t budget = pool_budget_words();
        int64_t most = words_big + words_small;
        if (n_act > 0 && most <= budget) {
            groups.emplace_back(0, n_act);
        } else if (n_act > 0) {
            // pool words in heavy-first order, prefix sums, groups
            cum.assign(n_act + 1, 0);
            DevBuf<int64_t> dcum(n_act + 1, s);
            k_gather_words<<<grid_for(n_act + 1, B), B, 0, s>>>(order, dprime, rsv_c, n_act, dcum.ptr);
            SBC_LAUNCHED();
            g_launches++;
            scan_exclusive_i64(dcum.ptr, dcum.ptr, n_act + 1, nullptr, s);
            SBC_CUDA(cudaMemcpyAsync(cum.data(), dcum.ptr, 8 * (size_t)(n_act + 1),
                                     cudaMemcpyDeviceToHost, s));
            SBC_CUDA(cudaStreamSynchronize(s));
            most = 1;
            for (int64_t a = 0; a < n_act;) {
                int64_t b = std::upper_bound(cum.begin() + a + 1, cum.end(), cum[a] + budget) -
                            cum.begin() - 1;
                if (b <= a) b = a + 1;  // one anchor larger than the budget runs alone
                groups.emplace_back(a, b);
                most = std::max(most, cum[b] - cum[a]);
                a = b;
            }
            cum_dev = std::move(dcum);
        }
        several = groups.size() > 1;
        pool.alloc((size_t)std::max<int64_t>(most, 1), s);
        const int sms = sm_count();

        ta.A_off = o->A_off.ptr;
        ta.A_ent = o->A_ent.ptr;
        ta.A_pos = o->A_pos.ptr;
        ta.A_bit = A_bit;
        ta.B_off = o->B_off.ptr;
        ta.B_ent = o->B_ent.ptr;
        ta.dprime = dprime;
        ta.e_use = e_use;
        ta.e_all = e_all;
        ta.rsv_c = rsv_c;
        ta.pool_off = pool_off;
        ta.order = order;
        ta.pool = pool.ptr;
        ta.ncand = ncand;
        ta.npaper = npaper;
        ta.nrow = nrow;
        ta.rinfo = rinfo;
        ta.single = R == 1;
        ta.n_ranks = (uint32_t)nX;
        ta.cnt = cnt.ptr;
        ta.l = l;
        ta.check = spec.check ? 1 : 0;
        ta.hs_cap = hash_slots_cap();
        ta.wcap = twohop_window_wedges();
        ta.bucket = nullptr;
        ta.bucket_slot = 0;
        if (hc.n_direct > 0) {
            const void *fn = spec.check ? (const void *)k_twohop_direct<true> : (const void *)k_twohop_direct<false>;
            gd = sms * blocks_per_sm(fn, DT_THREADS, DT_SMEM);
        }
        if (hc.n_big > 0) {
            const void *fn = spec.paper ? (const void *)k_twohop_large<true> : (const void *)k_twohop_large<false>;
            ga = sms * blocks_per_sm(fn, PL_THREADS, PL_SMEM);
            if ((int64_t)ga > (int64_t)hc.n_big) ga = (int)hc.n_big;
            // (reserved for every CTA-wide anchor: what a call needs does not
            // depend on the strategy its anchors take)
            if (hc.e_max > (unsigned long long)ta.wcap) {
                const int lgb = bucket_lg(hc.e_max);
                ta.bucket_slot = bucket_cap(hc.e_max, lgb) << lgb;
                bucket.alloc((size_t)ga * ta.bucket_slot, s);
                ta.bucket = bucket.ptr;
            }
        }
        if (hc.n_active > hc.n_big) {
            const void *fn = spec.paper ? (const void *)k_twohop_small<true> : (const void *)k_twohop_small<false>;
            gs = sms * blocks_per_sm(fn, PS_THREADS, PS_SMEM);
        }
        const int gb = sms;  // one tuple CTA per SM (its shared memory)
        const uint32_t wmax = (uint32_t)((o->max_deg_x + 31) / 32);
        per.alloc(spec.per_anchor ? 2 * nX : 0, s);
        if (per.ptr) SBC_CUDA(cudaMemsetAsync(per.ptr, 0, per.bytes(), s));
        if (spec.per_graph) SBC_CUDA(cudaMemsetAsync(spec.per_graph, 0, 16 * (size_t)spec.n_graphs, s));
        // prefix masks of the widest anchors, where they do not fit the warp's shared area
        scratch.alloc(R > 2 && (uint64_t)(R - 1) * wmax > TU_LIST_W
                          ? (size_t)gb * TU_WARPS * SCRATCH_SLOTS * wmax : 0, s);
        Totals tot;
        tot.total = cnt.ptr->total;
        tot.per_anchor = per.ptr;
        tot.per_graph = spec.per_graph;
        tot.graph_x0 = spec.graph_x0;
        tot.n_graphs = spec.n_graphs;
        tot.err = &cnt.ptr->err;
        ta.tot = tot;
        tu.nrow = nrow;
        tu.dprime = dprime;
        tu.rsv_c = rsv_c;
        tu.pool_off = pool_off;
        tu.pool = pool.ptr;
        tu.cnt = cnt.ptr;
        tu.tot = tot;
        tu.wide_scratch = scratch.ptr;
        tu.wmax = wmax;
        tu.l = l;

        ItemArgs ia;
        ia.ncand = ncand;
        ia.npaper = npaper;
        ia.nrow = nrow;
        ia.dprime = dprime;
        ia.rsv_c = rsv_c;
        ia.pool_off = pool_off;
        ia.rinfo = rinfo;
        ia.order = order;
        ia.R = R;
        ia.l = l;
        ia.method = spec.method;
        ia.pos_unit = (float)spec.pos_unit;
        ia.items_per_launch = 2.0f * (float)gb *
            (float)(spec.split_per_warp > 0 ? (unsigned long long)spec.split_per_warp : kSplitPerWarp);
        ia.cnt = cnt.ptr;
        ia.tc_on = spec.tc_min_w >= 0 && R == 2 && !thread_arena_active();
        ia.tc_min_w = spec.tc_min_w > 0 ? (uint32_t)spec.tc_min_w : kTcMinWords;
        ia.tc_min_nc = tc_min_candidates();
        if (ia.tc_on) tc_ensure_attrs();
        tc_plans.clear();
        tc_plans.resize(groups.size());
        n_items = 0;
        for (size_t gi = 0; gi < groups.size(); gi++) {
            const int64_t a = groups[gi].first, b = groups[gi].second, na = b - a;
            if (!cum.empty()) {
                // this group's pool offsets and fresh queue heads
                k_group_offsets<<<grid_for(na, B), B, 0, s>>>(order, cum_dev.ptr, a, b, pool_off);
                SBC_LAUNCHED();
                g_launches++;
                SBC_CUDA(cudaMemsetAsync(&cnt.ptr->head_direct, 0, 5 * sizeof(unsigned), s));
                SBC_CUDA(cudaMemsetAsync(&cnt.ptr->cost_total, 0,
                                         offsetof(Counters, run_begin) - offsetof(Counters, cost_total), s));
                SBC_CUDA(cudaMemsetAsync(&cnt.ptr->tw_fin_max, 0, 2 * sizeof(unsigned long long), s));
            }
            cudaEvent_t t0 = timing ? new_event(ev_twohop) : nullptr;
            cudaEvent_t t1 = timing ? new_event(ev_twohop) : nullptr;
            zero_pool(gi);
            if (t0) SBC_CUDA(cudaEventRecord(t0, s));
            {
                NvtxRange nr("sbc/twohop");
                launch_twohop((unsigned)a, (unsigned)b);
            }
            if (t1) SBC_CUDA(cudaEventRecord(t1, s));
            // tuple phase planning (needs the row counts)
            ia.begin = a;
            ia.nX = na;
            k_anchor_cost<<<grid_for(na, B), B, 0, s>>>(ia);
            SBC_LAUNCHED();
            g_launches++;
            if (R == 1) continue;  // the 2-hop kernels added every sum
            // room for the most items there can be (k_items), so that nothing
            // has to be read back first
            const size_t split = (size_t)ia.items_per_launch + 64;
            items.alloc((size_t)na + split, s);
            warp_list.alloc((size_t)na, s);
            claims.alloc(split, s);
            tc_in.alloc(ia.tc_on ? (size_t)na : 0, s);
            ia.items = items.ptr;
            ia.warp_list = warp_list.ptr;
            ia.tc_in = tc_in.ptr;
            SBC_CUDA(cudaMemsetAsync(claims.ptr, 0, claims.bytes(), s));
            k_items<<<grid_for(na, B), B, 0, s>>>(ia);
            SBC_LAUNCHED();
            g_launches++;
            std::vector<TcInput> tci;
            if (ia.tc_on) {
                // the listed anchors are planned on the host while the tuple
                // kernel runs; the first of them come with the counters
                tci.resize(std::min<size_t>((size_t)na, 2048));
                SBC_CUDA(cudaMemcpyAsync(tci.data(), tc_in.ptr, sizeof(TcInput) * tci.size(),
                                         cudaMemcpyDeviceToHost, s));
                SBC_CUDA(cudaMemcpyAsync(&hc, cnt.ptr, sizeof(Counters), cudaMemcpyDeviceToHost, s));
                SBC_CUDA(cudaStreamSynchronize(s));
                const size_t have = tci.size();
                tci.resize(hc.n_tc);
                if (tci.size() > have) {
                    SBC_CUDA(cudaMemcpyAsync(tci.data() + have, tc_in.ptr + have,
                                             sizeof(TcInput) * (tci.size() - have), cudaMemcpyDeviceToHost, s));
                    SBC_CUDA(cudaStreamSynchronize(s));
                }
            }
            tu.items = items.ptr;
            tu.warp_list = warp_list.ptr;
            tu.claims = claims.ptr;
            gt = (int)std::min<int64_t>(gb, na);
            if (ia.tc_on && hc.n_items == 0 && hc.n_warp == 0) gt = 0;
            if (gt > 0) {
                cudaEvent_t t2 = timing ? new_event(ev_tuples) : nullptr;
                cudaEvent_t t3 = timing ? new_event(ev_tuples) : nullptr;
                if (t2) SBC_CUDA(cudaEventRecord(t2, s));
                {
                    NvtxRange nr("sbc/tuples");
                    launch_tuple_kernel();
                }
                if (t3) SBC_CUDA(cudaEventRecord(t3, s));
            }
            if (!tci.empty()) plan_tc(gi, tci);
            run_tc_timed(gi, timing);
            if (!cum.empty()) {  // a further group clears the counters
                SBC_CUDA(cudaMemcpyAsync(&hc, cnt.ptr, sizeof(Counters), cudaMemcpyDeviceToHost, s));
                SBC_CUDA(cudaStreamSynchronize(s));
                tw_tail_ms = std::max(tw_tail_ms, group_tail_ms());
                n_items += hc.n_items + hc.n_warp;
            }
        }
        if (tm) tm->mark(4, s);
        collect();
        if (timing) {
            ms_twohop = pairs_ms(ev_twohop);
            ms_tuples = pairs_ms(ev_tuples);
            ms_tc = pairs_ms(ev_tc);
        }
        if (cum.empty()) res.work_items = (uint64_t)hc.n_items + hc.n_warp;
    }

    // Read the counters after an execution (synchronises the stream).
    void collect() {
        SBC_CUDA(cudaMemcpyAsync(&hc, cnt.ptr, sizeof(Counters), cudaMemcpyDeviceToHost, s));
        SBC_CUDA(cudaStreamSynchronize(s));
        if (hc.err & CERR_OVERFLOW) fail(SBC_E_OVERFLOW, "balanced biclique count exceeds 128 bits");
        if (hc.err & CERR_MASK)
            fail(SBC_E_CUDA, "self-check failed: a candidate mask disagrees with its 2-hop "
                             "counters (flags 0x%x)", hc.err);
        if (hc.err & CERR_TIMEOUT)
            fail(SBC_E_TIMEOUT, "a bounded wait of the tensor-core pair kernel ran out (flags 0x%x)",
                 hc.err);
        if (hc.err & (CERR_RESERVE | CERR_HASH))
            fail(SBC_E_CUDA, "internal error in the 2-hop kernel (flags 0x%x)", hc.err);
        res.count.lo = hc.total[0];
        res.count.hi = hc.total[1];
        const unsigned long long *tt = spec.paper ? hc.tuples_paper : hc.tuples_ours;
        res.anchor_tuples.lo = tt[0];
        res.anchor_tuples.hi = tt[1];
        res.candidates = hc.candidates;
        res.wedges = hc.wedges;
        if (!cum.empty()) res.work_items = (uint64_t)n_items;
        res.tested = hc.tested;
        res.typed = hc.leaves;
        res.popc_words = hc.popc_words;
        res.tc_anchors = tc_anchors;
        res.tc_tiles = tc_tiles;
        res.tc_kblocks = tc_kblocks;
        res.twohop_reads = hc.tw_reads;
        res.twohop_split = hc.tw_split;
        const double cyc = (double)(hc.tw_cyc[0] + hc.tw_cyc[1] + hc.tw_cyc[2] + hc.tw_cyc[3]);
        for (int i = 0; i < 4; i++) {
            res.twohop_anchors[i] = hc.tw_anchors[i];
            res.twohop_share[i] = cyc > 0 ? (float)(hc.tw_cyc[i] / cyc) : 0.f;
        }
        res.twohop_tail_ms = std::max(tw_tail_ms, group_tail_ms());
        res.pool_bytes = (uint64_t)(words_big + words_small) * 4;
    }
};

CountRun *countrun_create(const Orient &o, int64_t nnz, const CountSpec &spec, cudaStream_t s,
                          EventTimer *tm) {
    if (o.max_deg_x >= (1ll << 21))
        fail(SBC_E_UNSUPPORTED, "anchor-side degree %lld exceeds the 2^21 - 1 limit of the 2-hop counters",
             (long long)o.max_deg_x);
    ensure_kernel_attrs();
    std::unique_ptr<CountRun> run(new CountRun());
    run->o = &o;
    run->nnz = nnz;
    run->nX = o.nX;
    run->spec = spec;
    run->s = s;
    if (nnz > 0 && o.nX > 0) run->plan_and_run(tm);
    return run.release();
}

const CountResult &countrun_result(const CountRun *r) { return r->res; }

void countrun_launch(CountRun *r, cudaStream_t s) {
    if (r->nnz == 0 || r->nX == 0) {
        if (r->spec.per_graph) SBC_CUDA(cudaMemsetAsync(r->spec.per_graph, 0, 16 * (size_t)r->spec.n_graphs, s));
        return;
    }
    cudaStream_t keep = r->s;
    r->s = s;
    if (r->several) {
        // a multi-group plan re-plans (host reads between groups)
        cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
        SBC_CUDA(cudaStreamIsCapturing(s, &cs));
        if (cs != cudaStreamCaptureStatusNone) {
            r->s = keep;
            fail(SBC_E_UNSUPPORTED, "a count planned in %zu anchor groups cannot be captured",
                 r->groups.size());
        }
        try {
            r->plan_and_run(nullptr);
        } catch (...) {
            // the blocks stay with the plan and may next be freed on another stream
            (void)cudaStreamSynchronize(s);
            r->s = keep;
            throw;
        }
    } else {
        r->launch_count();
    }
    r->s = keep;
}

bool countrun_replayable(const CountRun *r) { return !r->several; }

void countrun_collect(CountRun *r, cudaStream_t s) {
    if (r->nnz == 0 || r->nX == 0) return;
    cudaStream_t keep = r->s;
    r->s = s;
    r->collect();
    r->s = keep;
}

void countrun_destroy(CountRun *r) { delete r; }

void apply_tune(CountSpec &spec, const sbc_tune_t *t) {
    if (!t) return;
    if (t->small_wedges < 0 || t->small_wedges > SMALL_E_MAX)
        fail(SBC_E_INVAL, "small_wedges must be in [0, %d], got %d", SMALL_E_MAX, t->small_wedges);
    if (t->pos_node_cost < 0 || t->pos_node_cost > (1 << 20))
        fail(SBC_E_INVAL, "pos_node_cost must be in [0, 2^20], got %d", t->pos_node_cost);
    if (t->split_per_warp < 0 || t->split_per_warp > 64)
        fail(SBC_E_INVAL, "split_per_warp must be in [0, 64], got %d", t->split_per_warp);
    if (t->tc_min_words < -1 || t->tc_min_words > 65536)
        fail(SBC_E_INVAL, "tc_min_words must be in [-1, 65536], got %d", t->tc_min_words);
    if (t->small_wedges) spec.small_e = t->small_wedges;
    if (t->pos_node_cost) spec.pos_unit = (unsigned long long)t->pos_node_cost;
    if (t->split_per_warp) spec.split_per_warp = t->split_per_warp;
    if (t->tc_min_words) spec.tc_min_w = t->tc_min_words;
}

// SBC_HASH_SLOTS_CAP (tests only): caps every 2-hop hash table at this many
// slots (rounded down to a multiple of 32, at least 32) so that tables
// overflow and the kernels' CERR_HASH report can be exercised.
uint32_t hash_slots_cap() {
    const char *e = getenv("SBC_HASH_SLOTS_CAP");
    if (!e || !*e) return 0;
    long long v = atoll(e);
    if (v <= 0) return 0;
    if (v > (1 << 20)) v = 1 << 20;
    v &= ~31ll;
    return (uint32_t)(v < 32 ? 32 : v);
}

// Visited wedges up to which the CTA-wide 2-hop kernel hashes an anchor in one
// window (above: bucketed by hash class). SBC_TWOHOP_WINDOW (tests only)
// lowers it, from 32 up, so that small graphs take the bucketed strategy.
uint32_t twohop_window_wedges() {
    const char *e = getenv("SBC_TWOHOP_WINDOW");
    long long v = e && *e ? atoll(e) : 0;
    if (v <= 0 || v > PL_WCAP) return (uint32_t)PL_WCAP;
    return (uint32_t)(v < 32 ? 32 : v);
}

// Candidates an anchor needs for the tensor-core pair step (tuning override
// SBC_TC_MIN_CANDIDATES, at least 2).
uint32_t tc_min_candidates() {
    uint32_t v = kTcMinCandidates;
    if (const char *e = getenv("SBC_TC_MIN_CANDIDATES")) {
        long long x = atoll(e);
        if (x >= 2 && x < (1ll << 31)) v = (uint32_t)x;
    }
    return v;
}

bool debug_checks_env() {
    const char *e = getenv("SBC_DEBUG");
    return e && *e && *e != '0';
}

unsigned long long pos_node_cost_setting() {
    unsigned long long u = kPosNodeCost;
    if (const char *e = getenv("SBC_POS_NODE_COST")) {  // tuning override
        long long v = atoll(e);
        if (v > 0) u = (unsigned long long)v;
    }
    return u;
}

void count_graph(const sbc_graph *gc, int p, int q, const sbc_count_opts *opts,
                 sbc_count_stats *stats, cudaStream_t s, bool timing) {
    sbc_graph *g = const_cast<sbc_graph *>(gc);
    if (p < 2 || q < 2 || p > 8 || q > 8) fail(SBC_E_INVAL, "p and q must be in [2, 8], got (%d, %d)", p, q);
    int cur = 0;
    SBC_CUDA(cudaGetDevice(&cur));
    if (cur != g->device) fail(SBC_E_INVAL, "graph lives on device %d, current device is %d", g->device, cur);
    int side = opts ? opts->anchor_side : SBC_SIDE_AUTO;
    if (side == SBC_SIDE_AUTO) side = preferred_side(g, p, q);
    if (side != 0 && side != 1) fail(SBC_E_INVAL, "anchor_side must be -1, 0 or 1");
    CountSpec spec;
    spec.k = side == 0 ? p : q;
    spec.l = side == 0 ? q : p;
    spec.paper = opts && (opts->flags & SBC_COUNT_PAPER_TUPLES);
    spec.shard = opts ? opts->shard : 0;
    spec.nshard = opts ? opts->shard_count : 0;
    spec.method = (opts && (opts->flags & SBC_COUNT_CANDIDATE_SIDE)) ? 1
                : (opts && (opts->flags & SBC_COUNT_POSITION_SIDE)) ? 2 : 0;
    spec.pos_unit = pos_node_cost_setting();
    apply_tune(spec, opts ? opts->tune : nullptr);
    spec.per_anchor = opts && opts->per_anchor;
    spec.check = (opts && (opts->flags & SBC_COUNT_CHECK)) || debug_checks_env();
    if (spec.nshard < 0 || (spec.nshard > 0 && (spec.shard < 0 || spec.shard >= spec.nshard)))
        fail(SBC_E_INVAL, "bad shard %d of %d", spec.shard, spec.nshard);
    const int64_t kernels0 = g_launches.load();
    if (stats) {
        memset(stats, 0, sizeof(*stats));
        stats->anchor_side = side;
    }
    const int64_t nX = side == 0 ? g->n_u : g->n_v;
    if (opts && opts->per_anchor && nX > 0) memset(opts->per_anchor, 0, sizeof(sbc_u128) * (size_t)nX);
    if (g->nnz == 0 || nX == 0) return;
    EventTimer tm(timing && stats != nullptr && !thread_arena_active());
    tm.mark(0, s);
    {
        std::lock_guard<std::mutex> lock(g->mu);
        NvtxRange nr("sbc/orientation");
        build_orientation(g, side, s);
    }
    const Orient &o = g->side[side];
    std::unique_ptr<CountRun> run(countrun_create(o, g->nnz, spec, s, tm.on ? &tm : nullptr));
    const CountResult &res = run->res;
    if (spec.per_anchor && run->per.ptr) {
        std::vector<unsigned long long> hp((size_t)2 * nX);
        std::vector<int32_t> vo((size_t)nX);
        SBC_CUDA(cudaMemcpyAsync(hp.data(), run->per.ptr, run->per.bytes(), cudaMemcpyDeviceToHost, s));
        SBC_CUDA(cudaMemcpyAsync(vo.data(), o.vert_of.ptr, (size_t)nX * 4, cudaMemcpyDeviceToHost, s));
        SBC_CUDA(cudaStreamSynchronize(s));
        for (int64_t r = 0; r < nX; r++) {
            opts->per_anchor[vo[r]].lo = hp[2 * r];
            opts->per_anchor[vo[r]].hi = hp[2 * r + 1];
        }
    }
    if (stats) {
        stats->count = res.count;
        stats->anchor_tuples = res.anchor_tuples;
        stats->candidates = res.candidates;
        stats->wedges = res.wedges;
        stats->work_items = res.work_items;
        stats->tuples_tested = res.tested;
        stats->tuples_typed = res.typed;
        stats->popc_words = res.popc_words;
        stats->tc_anchors = res.tc_anchors;
        stats->tc_tiles = res.tc_tiles;
        stats->tc_kblocks = res.tc_kblocks;
        stats->twohop_reads = res.twohop_reads;
        stats->twohop_split_classes = res.twohop_split;
        for (int i = 0; i < 4; i++) {
            stats->twohop_anchors[i] = res.twohop_anchors[i];
            stats->twohop_share[i] = res.twohop_share[i];
        }
        stats->twohop_tail_ms = res.twohop_tail_ms;
        stats->pool_bytes = res.pool_bytes;
        stats->kernels = (int32_t)(g_launches.load() - kernels0);
        if (tm.on) {
            stats->ms_total = tm.ms(0, 4);
            stats->ms_twohop = run->ms_twohop;
            stats->ms_tuples = run->ms_tuples;
            stats->ms_tc = run->ms_tc;
            stats->ms_prepare = stats->ms_total - run->ms_twohop - run->ms_tuples - run->ms_tc;
        }
    }
}

}  // namespace sbc
