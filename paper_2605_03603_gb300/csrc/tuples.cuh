// Tuple step (Algorithm 2, the loop over (p-1)-subsets A of C, and the type
// count of Section 4.2) over part rows; included once, by count.cu, inside
// its anonymous namespace.
//
// The 2-hop step leaves, per anchor, n rows of W mask words: one row per
// candidate c and part (same sign S_c = P_c & ~D_c, different sign
// T_c = P_c & D_c) that holds at least l positions. By Lemma 1 and its
// converse a type class of a tuple is the intersection of one part per
// partner, and the two parts of one candidate are disjoint, so
//   sum over R-subsets A of C, types k of binom(x[k], l)
//     = sum over R-subsets of rows of binom(|intersection|, l)          (1)
//     = sum over l-subsets Q of positions of binom(N_Q, R),             (2)
// N_Q = number of rows that contain Q. Two enumerations share one kernel:
//
// * rows (1): the rows are taken in ascending popcount; for every first row a
//   the later rows that share at least l positions with it are listed and
//   projected onto a's positions, so the remaining levels run on
//   ceil(|a| / 32) words (one, for most rows) instead of W. Bound by the latency
//   of AND, POPC and table lookup with four warps per scheduler (56 % of the issue
//   slots, POPC pipe 22 % on the (4,4) count of the 500k-edge graph).
// * column masks (2): for dense rows and few positions, a warp walks the
//   position subsets depth first over the bitmaps "rows that hold position q",
//   dropping prefixes contained in fewer than R rows.
// (Counting every row's l-subsets of positions in shared-memory counters, the
// third way to evaluate (2), was measured on the 2M-edge graph: (4,4) 231 ms
// against 107 for the rows, (3,3) 3.2 against 1.7; the counters of a window are
// too sparse to pay for clearing them.)
#pragma once

// ------------------------------------------------------------------ planning

// Saturating binom(n, k) in 64 bits (reported tuple counts and planning).
__device__ __forceinline__ unsigned long long binom_sat(unsigned long long n, int k) {
    if ((long long)n < k) return 0;
    unsigned long long r = 1;
    for (int i = 1; i <= k; i++) {
        unsigned long long f = n - k + i;
        if (r > 0xFFFFFFFFFFFFFFFFull / f) return 0xFFFFFFFFFFFFFFFFull;
        r = r * f / i;
    }
    return r;
}

// A work item: first rows (or, with cols, first positions of the column walk)
// of the anchor, claimed from the shared counter `claim` by every item of the
// anchor (NO_CLAIM: the anchor has one item).
struct Item {
    uint32_t anchor, claim, cols;
};
constexpr uint32_t NO_CLAIM = 0xFFFFFFFFu;

constexpr int TU_THREADS = 512;
constexpr int TU_WARPS = TU_THREADS / 32;
constexpr uint32_t TU_ROWS_W = 20480;             // staged row words (80 KB)
constexpr uint32_t TU_LIST_W = 1536;              // words of a warp's list (6 KB)
constexpr uint32_t TU_LISTS_W = TU_LIST_W * TU_WARPS;
constexpr uint32_t TU_BUF_N = 64;                 // prefixes a warp collects, of up to 4 words
constexpr uint32_t TU_BUF_W = TU_BUF_N * 5;
constexpr uint32_t TU_PERM = 8192;                // rows of an ordered anchor
constexpr uint32_t TU_OFF_LIST = TU_ROWS_W;
constexpr uint32_t TU_OFF_BUF = TU_ROWS_W + TU_LISTS_W;
constexpr uint32_t TU_OFF_PERM = TU_OFF_BUF + TU_BUF_W * TU_WARPS;
constexpr size_t TU_SMEM = (size_t)(TU_OFF_PERM + TU_PERM / 2) * 4;
constexpr uint32_t CW_MAX_WORDS = 128;            // row words of a column mask (4 per lane)
// A prefix node of the column walk costs CW_NODE * pos_node_cost mask words per
// 32 row words. The 20k-edge graph's (5,5) took 1.6 / 0.67 / 0.40 / 0.40 ms and
// its (5,7) 3.1 / 1.8 / 1.8 / 3.2 ms at a product of 3 / 10 / 25 / 60.
constexpr float CW_NODE = 8.0f;

// Anchors this small are taken one per warp.
constexpr uint32_t WG_WORDS = 1024, WG_ROWS = 512;
constexpr int SCRATCH_SLOTS = 7;                  // per-warp prefix masks of the widest anchors

struct ItemArgs {
    const uint32_t *ncand, *npaper, *nrow, *dprime;
    RowInfo *rinfo;          // per anchor, set when it has rows; k_anchor_cost leaves its plan here
    const uint32_t *order;   // anchors of the group: order[begin .. begin + nX)
    int64_t begin;
    int64_t nX;              // anchors in the group
    int R, l;
    int method;  // 0: cheaper side per anchor, 1: rows, 2: column walk where it fits
    float pos_unit;
    float items_per_launch;  // items that the anchors' total cost is split into
    const uint32_t *rsv_c;
    const int64_t *pool_off;
    Item *items;             // room for nX + items_per_launch
    uint32_t *warp_list;     // ... nX
    Counters *cnt;
    // tensor-core pair step (two partners)
    int tc_on;
    uint32_t tc_min_w, tc_min_nc;
    TcInput *tc_in;          // ... nX
};

// Costs in mask-word operations (one AND + POPC of the row side).
__device__ __forceinline__ float rows_cost(float n, float dp, float pops, int R, int l) {
    const float W = ceilf(dp * (1.0f / 32.0f));
    float c = 0.5f * n * n * W;                    // first-level filter (all pairs)
    if (R > 2) {
        // later rows that survive the filter: about a fifth on power-law
        // graphs (CPU replay; rows share popular positions), all of them when
        // rows are dense enough to share l positions on average
        const float pbar = pops / n;
        const float m = fminf(fmaxf(pbar * pbar / (dp * (float)l), 0.2f), 1.0f) * n;
        float t = n * ceilf(pbar * (1.0f / 32.0f));
        for (int i = 2; i <= R; i++) t *= m / (float)i;
        c += t;
    }
    return c;
}

// An anchor's path, and the cost of its items (row and column paths). Kept in its
// RowInfo (the cost in place of the positions, the path above the longest row) from
// k_anchor_cost on, so that the items are made of the very costs that were totalled:
// the room for them rests on that.
enum : uint32_t { PATH_NONE = 0, PATH_TC = 1, PATH_WARP = 2, PATH_ROWS = 3, PATH_COLS = 4 };
constexpr int PATH_SHIFT = 28;  // (rows have fewer than 2^21 positions)
struct AnchorPlan {
    float cost = 0;
    uint32_t path = PATH_NONE;
};

// Which path(s) an anchor's tuples take.
__device__ __forceinline__ AnchorPlan plan_anchor(const ItemArgs &a, uint32_t r) {
    AnchorPlan p;
    const uint32_t n = a.nrow[r], nc = a.ncand[r], dp = a.dprime[r];
    if (a.R == 1 || n < (uint32_t)a.R || nc < (uint32_t)a.R) return p;
    const uint32_t W = (dp + 31) / 32;
    const float rc = rows_cost((float)n, (float)dp, a.rinfo[r].pops, a.R, a.l);
    const bool tc_ok = a.tc_on && a.R == 2 && nc >= a.tc_min_nc && W >= a.tc_min_w;
    // a 128 x 256 x 128 tensor-core step costs about as much as 1024 word operations
    const float tcc = 0.5f * (float)n * (float)n * (float)((W + 3) / 4) / 32.0f + 2048.0f;
    const float alt = tc_ok ? fminf(tcc, rc) : rc;
    if (a.method != 1) {
        // column walk: every prefix of up to l positions (before pruning),
        // 32 children at a time
        float cc = 3.0e38f;
        const uint32_t wc = (n + 31) / 32;
        if (dp >= (uint32_t)a.l && wc <= CW_MAX_WORDS && (unsigned long long)dp * (wc | 1u) <= TU_OFF_PERM) {
            float nodes = 0, t = 1;
            for (int i = 1; i <= a.l; i++) {
                t *= (float)(dp + 1 - i) / (float)i;
                nodes += t;
            }
            cc = nodes * CW_NODE * a.pos_unit * (float)((wc + 31) / 32);
        }
        if (cc < 3.0e38f && (a.method == 2 || cc < alt)) {
            p.path = PATH_COLS;
            p.cost = cc;
            return p;
        }
    }
    if (tc_ok) {
        p.path = PATH_TC;
    } else if (n * W <= WG_WORDS && n <= WG_ROWS && W <= 4 && rc <= 65536.0f) {
        p.path = PATH_WARP;
    } else {
        p.path = PATH_ROWS;
        p.cost = rc;
    }
    return p;
}

// Reported tuple counts, every anchor's plan, and the cost total that sizes the work items.
__global__ void k_anchor_cost(ItemArgs a) {
    U128 tp, to;
    unsigned long long cand = 0;
    double cost = 0;
    for (int64_t ix = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; ix < a.nX;
         ix += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t r = a.order[a.begin + ix];
        uint32_t nc = a.ncand[r];
        if (a.npaper) {
            uint32_t np = a.npaper[r];
            cand += np;
            if (np >= (uint32_t)a.R) {
                // binom(np, R) exactly: np < 2^32, R <= 7, fits 128 bits
                unsigned long long lo = 1, hi = 0;
                for (int i = 1; i <= a.R; i++) {
                    unsigned long long f = np - a.R + i;
                    unsigned g = gcd_u32((unsigned)(f % (unsigned)i), (unsigned)i);
                    if (g == 0) g = i;
                    div_u128_small(lo, hi, i / g);
                    mul_u128_u64(lo, hi, f / g);
                }
                U128 t;
                t.lo = lo;
                t.hi = hi;
                tp.add(t);
            }
        } else {
            cand += nc;
        }
        if (nc >= (uint32_t)a.R) to.add(binom_sat(nc, a.R));
        if (a.R > 1) {
            const AnchorPlan p = plan_anchor(a, r);
            a.rinfo[r].pops = p.cost;
            a.rinfo[r].longest |= p.path << PATH_SHIFT;
            cost += (double)p.cost;
        }
    }
    tp = warp_sum_u128(tp, nullptr);
    to = warp_sum_u128(to, nullptr);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        cand += __shfl_xor_sync(FULL, cand, o);
        cost += __shfl_xor_sync(FULL, cost, o);
    }
    if ((threadIdx.x & 31) == 0) {
        atomic_add_u128(a.cnt->tuples_paper, tp.lo, tp.hi, nullptr);
        atomic_add_u128(a.cnt->tuples_ours, to.lo, to.hi, nullptr);
        if (cand) atomicAdd(&a.cnt->candidates, cand);
        if (cost > 0) atomicAdd(&a.cnt->cost_total, cost);
    }
}

// Work items, warp list and tensor-core list of every anchor. An anchor's items
// depend on its sizes and the cost total only (a few operations per anchor: how
// its first rows are shared among its items is settled while they run). The
// items beyond one per anchor sum to at most items_per_launch: an anchor of
// several has at most cost / item_cost of them, the costs sum to cost_total, and the
// roundings (2^-22 of the sum together) cannot make another whole item.
__global__ void k_items(ItemArgs a) {
    const float item_cost = fmaxf((float)(a.cnt->cost_total / (double)a.items_per_launch), 16384.0f);
    for (int64_t ix = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; ix < a.nX;
         ix += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t r = a.order[a.begin + ix];
        const RowInfo info = a.rinfo[r];
        const uint32_t path = info.longest >> PATH_SHIFT;
        if (path == PATH_TC) {
            TcInput t;
            t.r = r;
            t.nr = a.nrow[r];
            t.W = (a.dprime[r] + 31) / 32;
            t.rsv = a.rsv_c[r];
            t.longest = info.longest & ((1u << PATH_SHIFT) - 1u);
            t.pool_off = a.pool_off[r];
            a.tc_in[atomicAdd(&a.cnt->n_tc, 1u)] = t;
        } else if (path == PATH_WARP) {
            a.warp_list[atomicAdd(&a.cnt->n_warp, 1u)] = r;
        } else if (path != PATH_NONE) {
            const uint32_t total = (uint32_t)fminf(fmaxf(info.pops / item_cost, 1.0f), 1024.0f);
            const unsigned k0 = atomicAdd(&a.cnt->n_items, total);
            const unsigned claim = total > 1 ? atomicAdd(&a.cnt->n_claims, 1u) : NO_CLAIM;
            for (uint32_t i = 0; i < total; i++) {
                Item it;
                it.anchor = r;
                it.claim = claim;
                it.cols = path == PATH_COLS;
                a.items[k0 + i] = it;
            }
        }
    }
}

// ------------------------------------------------------------------ kernel

struct TupleArgs {
    const uint32_t *nrow, *dprime, *rsv_c;
    const int64_t *pool_off;
    const uint32_t *pool;
    const Item *items;
    const uint32_t *warp_list;
    uint32_t *claims;
    Counters *cnt;
    Totals tot;
    uint32_t *wide_scratch;          // per warp: SCRATCH_SLOTS * wmax words, or null
    uint32_t wmax;
    int l;
};

// Per-lane tally: tuples whose common positions were counted, those with at
// least l, and the mask words popcounted for it.
struct Acc {
    U128 sum;
    unsigned long long tested = 0, leaves = 0, words = 0;
};

constexpr int BINOM_TBL = 256;

// Dynamic shared memory, and the table binom(x, l) for x <= BINOM_TBL
// (binom(256, 8) < 2^64).
extern __shared__ __align__(16) uint32_t sm_dyn[];
__shared__ unsigned long long s_bt[BINOM_TBL + 1];
__shared__ unsigned long long s_btR[BINOM_TBL + 1];  // binom(x, R), for the column walk
// binom(x, l) | leaf flag in 32 bits for the list loops: up to the x with
// 8 binom(x, l) < 2^27 eight entries sum without touching the flag bits, so
// one 32-bit add counts both the binomials and the tuples with x >= l.
constexpr int TBL32 = 128;
constexpr uint32_t LEAF = 1u << 27;
__shared__ uint32_t s_bt32[TBL32 + 1];
__shared__ uint32_t s_max32;  // largest x of s_bt32

// binom(x, K) with compile-time K.
template <int K>
__device__ __forceinline__ void binom_add_k(U128 &acc, unsigned long long x, unsigned *err) {
    if (x < (unsigned long long)K) return;
    if constexpr (K == 1) {
        acc.add(x);
    } else {
        if (x > c_binom64_max[K]) {
            if (acc.add(binom_slow(x, K, err))) atomicOr(err, CERR_OVERFLOW);
            return;
        }
        acc.add(binom_u64<K>(x));
    }
}

// Adds binom(n, l) of a closed tuple.
__device__ __forceinline__ void close_tuple(uint32_t n, int l, Acc &acc, unsigned *err) {
    if (n <= (uint32_t)BINOM_TBL) acc.sum.add(s_bt[n]);
    else binom_add(acc.sum, n, l, err);
    acc.leaves += n >= (uint32_t)l;
}

// An anchor's rows: staged in shared memory in row order (ST), or in the pool
// (word w of row i at g[w * stride + i]), ordered by perm when it is set.
template <bool ST>
struct RowsV {
    const uint32_t *g;
    const uint16_t *perm;
    uint32_t stride, W, n;
    __device__ __forceinline__ uint32_t word(uint32_t w, uint32_t i) const {
        if constexpr (ST) return sm_dyn[w * n + i];
        else return g[(size_t)w * stride + (perm ? (uint32_t)perm[i] : i)];
    }
};

// The last level of a list: prefixes of R - 1 rows collected from the level
// above, one per lane, each lane walking the entries after its own last one.
// (With the lanes over entries instead, a prefix of a short list leaves most
// of the warp idle and pays the loop's latency alone: the 20k-edge graph's
// (5,5) count took 1.3 ms that way.)
template <int WN>
struct PrefixBuf {
    uint32_t off, m, ms, W;  // the list: word w of entry i at sm_dyn[off + w * ms + i]
    uint32_t buf;            // sm_dyn index of the buffer
    uint32_t n = 0;          // prefixes in it (warp-uniform)

    __device__ __forceinline__ void close(uint32_t k0, uint32_t cnt, int l, Acc &acc) {
        const uint32_t lane = threadIdx.x & 31;
        uint32_t X[WN], c = m;
        const bool valid = lane < cnt;
#pragma unroll
        for (int w = 0; w < WN; w++) X[w] = valid && w < (int)W ? sm_dyn[buf + (1 + w) * TU_BUF_N + k0 + lane] : 0u;
        if (valid) c = sm_dyn[buf + k0 + lane];
        const uint32_t d0 = __reduce_min_sync(FULL, c) + 1;
        // counts <= 32 * WN <= 128: inside the table, zero below l; fewer than
        // 2^17 values below 2^41 fit 64 bits
        unsigned long long part = 0;
        uint32_t leaves = 0;
#pragma unroll 4
        for (uint32_t d = d0; d < m; d++) {
            uint32_t x = 0;
#pragma unroll
            for (int w = 0; w < WN; w++)
                if (w < (int)W) x += __popc(X[w] & sm_dyn[off + w * ms + d]);
            x = d > c ? x : 0u;
            part += s_bt[x];
            leaves += x >= (uint32_t)l;
        }
        acc.sum.add(part);
        acc.leaves += leaves;
        const uint32_t t = m - 1 - (c < m ? c : m - 1);
        acc.tested += t;
        acc.words += (unsigned long long)t * W;
    }
    // Lanes with `ok` add the prefix T whose last row is entry c.
    __device__ __forceinline__ void push(bool ok, const uint32_t (&T)[WN], uint32_t c, int l, Acc &acc) {
        const uint32_t lane = threadIdx.x & 31, bal = __ballot_sync(FULL, ok);
        if (!bal) return;
        if (ok) {
            const uint32_t k = n + __popc(bal & ((1u << lane) - 1u));
            sm_dyn[buf + k] = c;
#pragma unroll
            for (int w = 0; w < WN; w++)
                if (w < (int)W) sm_dyn[buf + (1 + w) * TU_BUF_N + k] = T[w];
        }
        n += __popc(bal);
        __syncwarp();
        if (n > TU_BUF_N - 32) {
            close(n - 32, 32, l, acc);
            n -= 32;
            __syncwarp();
        }
    }
    __device__ __forceinline__ void flush(int l, Acc &acc) {
        if (n) close(0, n, l, acc);
        n = 0;
        __syncwarp();
    }
};

// Extend a warp-uniform prefix mask (L - 1 rows) by the entries start..m-1 of
// a list, lanes over entries; W <= WN words. Prefixes of R - 1 rows go to the
// buffer.
template <int L, int R, int WN>
__device__ void expand(PrefixBuf<WN> &pb, const uint32_t (&pre)[WN], uint32_t start, int l, Acc &acc) {
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t m = pb.m;
    for (uint32_t mb = start; mb < m; mb += 32) {
        const uint32_t c = mb + lane;
        const bool valid = c < m;
        uint32_t T[WN], n = 0;
#pragma unroll
        for (int w = 0; w < WN; w++) {
            T[w] = (valid && w < (int)pb.W) ? (pre[w] & sm_dyn[pb.off + w * pb.ms + c]) : 0u;
            n += __popc(T[w]);
        }
        const bool ok = valid && (int)n >= l && (m - 1 - c) >= (uint32_t)(R - L);
        if constexpr (L == R - 1) {
            pb.push(ok, T, c, l, acc);
        } else {
            uint32_t bal = __ballot_sync(FULL, ok);
            while (bal) {
                const int s = __ffs(bal) - 1;
                bal &= bal - 1;
                uint32_t Ts[WN];
#pragma unroll
                for (int w = 0; w < WN; w++) Ts[w] = __shfl_sync(FULL, T[w], s);
                expand<L + 1, R, WN>(pb, Ts, mb + s + 1, l, acc);
            }
        }
    }
    if (start + lane < m) {
        const uint32_t t = (m - 1 - start - lane) / 32 + 1;
        acc.tested += t;
        acc.words += (unsigned long long)t * pb.W;
    }
}

// All pairs of a list's entries (three rows in all) in tiles: a lane keeps
// four entries, entries b are read once for them (four at a time when W is 1).
// Blocks of 128 entries c0 = first, first + step, ... as the later entry. Used
// while every count is at most s_max32. A pair costs an AND and a POPC per word
// (half a warp per cycle and SM) and a table lookup. Taking the counts from the
// warp matrix instruction instead (bits as fp16 or fp8, the same lookups) was
// slower: (4,4) of the 2M-edge graph 137 and 153 against 105 ms.
template <int WN>
__device__ __forceinline__ void list_pairs_tiled(uint32_t off, uint32_t m, uint32_t ms, uint32_t first,
                                                 uint32_t step, Acc &acc) {
    const uint32_t lane = threadIdx.x & 31;
    unsigned long long sum = 0;
    uint32_t leaves = 0;
    auto settle = [&](uint32_t part) {
        sum += part & (LEAF - 1);
        leaves += part / LEAF;
    };
    for (uint32_t c0 = first; c0 < m; c0 += step) {
        uint32_t C[4][WN];
#pragma unroll
        for (int k = 0; k < 4; k++) {
            const uint32_t c = c0 + lane + 32 * k;
#pragma unroll
            for (int w = 0; w < WN; w++) C[k][w] = c < m ? sm_dyn[off + w * ms + c] : 0u;
        }
        const bool half = c0 + 64 >= m;  // the upper two groups are empty
        for (uint32_t b = 0; b < c0; b += 4) {
            uint32_t B[4][WN];
#pragma unroll
            for (int w = 0; w < WN; w++) {
                const uint4 v = *reinterpret_cast<const uint4 *>(&sm_dyn[off + w * ms + b]);
                B[0][w] = v.x;
                B[1][w] = v.y;
                B[2][w] = v.z;
                B[3][w] = v.w;
            }
#pragma unroll
            for (int h = 0; h < 2; h++) {
                uint32_t part = 0;
#pragma unroll
                for (int j = 0; j < 2; j++)
#pragma unroll
                    for (int k = 0; k < 4; k++) {
                        if (k >= 2 && half) break;
                        uint32_t n = 0;
#pragma unroll
                        for (int w = 0; w < WN; w++) n += __popc(B[2 * h + j][w] & C[k][w]);
                        part += s_bt32[n];
                    }
                settle(part);
            }
        }
        // the block's own pairs: 32 earlier entries at a time against the
        // groups of 32 lanes that are not before them
        const uint32_t be = c0 + 128 < m ? c0 + 128 : m;
#pragma unroll
        for (int jb = 0; jb < 4; jb++) {
            const uint32_t b0 = c0 + 32 * jb;
            const uint32_t b1 = b0 + 32 < be ? b0 + 32 : be;
            for (uint32_t b = b0; b < b1; b++) {
                uint32_t part = 0;
#pragma unroll
                for (int k = jb; k < 4; k++) {
                    uint32_t n = 0;
#pragma unroll
                    for (int w = 0; w < WN; w++) n += __popc(sm_dyn[off + w * ms + b] & C[k][w]);
                    part += k > jb || b0 + lane > b ? s_bt32[n] : 0u;
                }
                settle(part);
            }
        }
        if (lane == 0) {
            const unsigned long long nb = be - c0, t = nb * c0 + nb * (nb - 1) / 2;
            acc.tested += t;
            acc.words += t * WN;
        }
    }
    acc.sum.add(sum);
    acc.leaves += leaves;
}

// Second and later rows of one first row: entries b = b0, b0 + step, ... of
// its list, W words each.
template <int R, int WN>
__device__ __forceinline__ void list_seconds(uint32_t off, uint32_t m, uint32_t ms, uint32_t W,
                                             uint32_t buf, uint32_t b0, uint32_t step, int l, Acc &acc) {
    PrefixBuf<WN> pb;
    pb.off = off;
    pb.m = m;
    pb.ms = ms;
    pb.W = W;
    pb.buf = buf;
    if constexpr (R == 3) {
        // a prefix of R - 1 rows is the first row and one entry
        for (uint32_t b = 32 * b0; b < m; b += 32 * step) {
            const uint32_t c = b + (threadIdx.x & 31);
            uint32_t T[WN];
#pragma unroll
            for (int w = 0; w < WN; w++) T[w] = c < m && w < (int)W ? sm_dyn[off + w * ms + c] : 0u;
            pb.push(c + 1 < m, T, c, l, acc);
        }
    } else {
        for (uint32_t b = b0; b + (R - 2) < m; b += step) {
            uint32_t pre[WN];
#pragma unroll
            for (int w = 0; w < WN; w++) pre[w] = w < (int)W ? sm_dyn[off + w * ms + b] : 0u;
            expand<3, R, WN>(pb, pre, b + 1, l, acc);
        }
    }
    pb.flush(l, acc);
}

// The same for three rows in all and lists of any width: words streamed.
__device__ __forceinline__ void list_pairs_wide(uint32_t off, uint32_t m, uint32_t ms, uint32_t W,
                                                uint32_t b0, uint32_t step, int l, Acc &acc,
                                                unsigned *err) {
    const int lane = threadIdx.x & 31;
    for (uint32_t b = b0; b + 1 < m; b += step)
        for (uint32_t c = b + 1 + lane; c < m; c += 32) {
            uint32_t n = 0;
            for (uint32_t w = 0; w < W; w++) n += __popc(sm_dyn[off + w * ms + b] & sm_dyn[off + w * ms + c]);
            close_tuple(n, l, acc, err);
            acc.tested++;
            acc.words += W;
        }
}

// The tuples of a list of m entries (plane stride ms, W words, at most `pa`
// positions), shared among `warps` warps.
template <int R>
__device__ __forceinline__ void list_all(uint32_t off, uint32_t m, uint32_t ms, uint32_t W, uint32_t pa,
                                         uint32_t wi, uint32_t warps, int l, Acc &acc, unsigned *err) {
    if constexpr (R == 3) {
        if (pa <= s_max32 && W == 1) return list_pairs_tiled<1>(off, m, ms, 128 * wi, 128 * warps, acc);
        if (pa <= s_max32 && W == 2) return list_pairs_tiled<2>(off, m, ms, 128 * wi, 128 * warps, acc);
    }
    const uint32_t buf = TU_OFF_BUF + (threadIdx.x >> 5) * TU_BUF_W;
    if (W == 1) list_seconds<R, 1>(off, m, ms, W, buf, wi, warps, l, acc);
    else if (W == 2) list_seconds<R, 2>(off, m, ms, W, buf, wi, warps, l, acc);
    else if (W <= 4) list_seconds<R, 4>(off, m, ms, W, buf, wi, warps, l, acc);
    else if constexpr (R == 3) list_pairs_wide(off, m, ms, W, wi, warps, l, acc, err);
}

// Positions of row a, whose first four words are in A (every lane gets the sum).
template <bool ST>
__device__ __forceinline__ uint32_t row_positions(const RowsV<ST> &v, uint32_t a, const uint32_t (&A)[4]) {
    uint32_t n = 0;
#pragma unroll
    for (int w = 0; w < 4; w++) n += __popc(A[w]);
    if (v.W > 4) {
        uint32_t x = 0;
        for (uint32_t w = 4 + (threadIdx.x & 31); w < v.W; w += 32) x += __popc(v.word(w, a));
        n += __reduce_add_sync(FULL, x);
    }
    return n;
}

// Positions shared by row a (words A when W <= WN, else read again) and row c.
template <int WN, bool ST>
__device__ __forceinline__ uint32_t shared_count(const RowsV<ST> &v, const uint32_t (&A)[WN],
                                                 uint32_t c) {
    uint32_t n = 0;
#pragma unroll
    for (int w = 0; w < WN; w++)
        if (w < (int)v.W) n += __popc(A[w] & v.word(w, c));
    return n;
}
template <bool ST>
__device__ __forceinline__ uint32_t shared_count_wide(const RowsV<ST> &v, uint32_t a, uint32_t c) {
    uint32_t n = 0;
#pragma unroll 4
    for (uint32_t w = 0; w < v.W; w++) n += __popc(v.word(w, a) & v.word(w, c));
    return n;
}

// Two rows in all: first row a with every later row, lanes over rows.
template <int WN, bool ST>
__device__ __forceinline__ void pairs_narrow(const RowsV<ST> &v, uint32_t a, int l, Acc &acc) {
    uint32_t A[WN];
#pragma unroll
    for (int w = 0; w < WN; w++) A[w] = w < (int)v.W ? v.word(w, a) : 0u;
    // counts <= 32 * WN <= 256: inside the table; binom(256, 8) < 2^49, so 2^14
    // of them fit 64 bits
    unsigned long long part = 0;
    uint32_t leaves = 0, tested = 0;
    for (uint32_t c0 = a + 1; c0 < v.n; c0 += 32u << 14) {
        const uint32_t c1 = v.n - c0 < 32u << 14 ? v.n : c0 + (32u << 14);
#pragma unroll 4
        for (uint32_t c = c0 + (threadIdx.x & 31); c < c1; c += 32) {
            const uint32_t n = shared_count<WN, ST>(v, A, c);
            part += s_bt[n];
            leaves += n >= (uint32_t)l;
            tested++;
        }
        acc.sum.add(part);
        part = 0;
    }
    acc.leaves += leaves;
    acc.tested += tested;
    acc.words += (unsigned long long)tested * v.W;
}
template <bool ST>
__device__ __forceinline__ void pairs_of(const RowsV<ST> &v, uint32_t a, int l, Acc &acc, unsigned *err) {
    if (v.W == 1) pairs_narrow<1, ST>(v, a, l, acc);
    else if (v.W == 2) pairs_narrow<2, ST>(v, a, l, acc);
    else if (v.W <= 4) pairs_narrow<4, ST>(v, a, l, acc);
    else if (v.W <= 8) pairs_narrow<8, ST>(v, a, l, acc);
    else
        for (uint32_t c = a + 1 + (threadIdx.x & 31); c < v.n; c += 32) {
            close_tuple(shared_count_wide<ST>(v, a, c), l, acc, err);
            acc.tested++;
            acc.words += v.W;
        }
}

// Rows of [cb, cb + 32) that share at least l positions with row a (ballot).
template <bool ST>
__device__ __forceinline__ uint32_t survivors(const RowsV<ST> &v, uint32_t a, const uint32_t (&A)[4],
                                              uint32_t cb, int l, Acc &acc) {
    const uint32_t c = cb + (threadIdx.x & 31);
    bool ok = false;
    if (c < v.n) {
        uint32_t n;
        if (v.W == 1) n = __popc(A[0] & v.word(0, c));
        else if (v.W <= 4) n = shared_count<4, ST>(v, A, c);
        else n = shared_count_wide<ST>(v, a, c);
        acc.tested++;
        acc.words += v.W;
        ok = (int)n >= l;
    }
    return __ballot_sync(FULL, ok);
}

// Row c's bits at row a's positions, packed: writes its ceil(|a| / 32) words
// to entry k of the list at off (m entries, plane stride ms). Lanes hold different c, the
// walk over a's bits is the warp's.
template <bool ST>
__device__ __forceinline__ void project_row(const RowsV<ST> &v, uint32_t a, uint32_t c, uint32_t off,
                                            uint32_t m, uint32_t ms, uint32_t k) {
    uint32_t out = 0, nb = 0, plane = 0;
    for (uint32_t w = 0; w < v.W; w++) {
        uint32_t aw = v.word(w, a);
        if (!aw) continue;
        const uint32_t x = v.word(w, c);
        while (aw) {
            const int b = __ffs(aw) - 1;
            aw &= aw - 1;
            out |= ((x >> b) & 1u) << nb;
            if (++nb == 32) {
                if (k < m) sm_dyn[off + plane * ms + k] = out;
                plane++;
                out = 0;
                nb = 0;
            }
        }
    }
    if (nb && k < m) sm_dyn[off + plane * ms + k] = out;
}

// The part of project_row that a's words [w0, w1) give, ORed into a list of zeros
// (several warps share the walk).
template <bool ST>
__device__ __noinline__ void project_words(const RowsV<ST> &v, uint32_t a, uint32_t c, uint32_t w0,
                                              uint32_t w1, uint32_t off, uint32_t m, uint32_t ms, uint32_t k) {
    uint32_t at = 0;  // position of the next bit
    for (uint32_t w = threadIdx.x & 31; w < w0; w += 32) at += __popc(v.word(w, a));
    at = __reduce_add_sync(FULL, at);
    uint32_t out = 0;
    uint32_t na = w0 < w1 ? v.word(w0, a) : 0u, nx = w0 < w1 ? v.word(w0, c) : 0u;
    for (uint32_t w = w0; w < w1; w++) {
        uint32_t aw = na;
        const uint32_t x = nx;
        if (w + 1 < w1) {
            na = v.word(w + 1, a);
            nx = v.word(w + 1, c);
        }
        while (aw) {
            const int b = __ffs(aw) - 1;
            aw &= aw - 1;
            out |= ((x >> b) & 1u) << (at & 31);
            if ((++at & 31) == 0) {
                if (k < m) atomicOr(&sm_dyn[off + (at / 32 - 1) * ms + k], out);
                out = 0;
            }
        }
    }
    if (out && k < m) atomicOr(&sm_dyn[off + (at / 32) * ms + k], out);
}

// ---- prefixes too wide for the lists: the prefix masks sit in the warp's
// list area (or its global scratch when they do not fit), every level tests
// the anchor's own rows.
template <int L, int R, bool ST>
__device__ __noinline__ void expand_wide(const RowsV<ST> &v, uint32_t *scr, uint32_t wstride,
                                         uint32_t start, uint32_t end, int l, Acc &acc, unsigned *err) {
    const int lane = threadIdx.x & 31;
    const uint32_t *pre = scr + (size_t)(L - 2) * wstride;  // L - 1 rows
    for (uint32_t mb = start; mb < end; mb += 32) {
        const uint32_t c = mb + lane;
        const bool valid = c < v.n;
        uint32_t n = 0;
        if (valid) {
            acc.tested++;
            acc.words += v.W;
            for (uint32_t w = 0; w < v.W; w++) n += __popc(pre[w] & v.word(w, c));
        }
        if constexpr (L == R) {
            if (valid && (int)n >= l) close_tuple(n, l, acc, err);
        } else {
            uint32_t bal = __ballot_sync(FULL, valid && (int)n >= l && (v.n - 1 - c) >= (uint32_t)(R - L));
            while (bal) {
                const uint32_t cs = mb + __ffs(bal) - 1;
                bal &= bal - 1;
                uint32_t *nxt = scr + (size_t)(L - 1) * wstride;
                __syncwarp();
                for (uint32_t w = lane; w < v.W; w += 32) nxt[w] = pre[w] & v.word(w, cs);
                __syncwarp();
                expand_wide<L + 1, R, ST>(v, scr, wstride, cs + 1, v.n, l, acc, err);
            }
        }
    }
}

constexpr uint32_t DEFER_MAX = 256;
// From this list length a first row of four or more rows in all is shared by
// the CTA's warps: its subtree grows with the third power or more (one warp
// alone held the 20k-edge graph's (5,5) count for 0.4 ms).
constexpr uint32_t CTA_LIST = 40;

struct TupleShared {
    unsigned item, unit, ndefer, m, n_units, words;
    uint32_t defer[DEFER_MAX];
    uint32_t hist[256];
};

// One first row on one warp. Lists that do not fit go to the CTA (defer).
template <int R, bool ST>
__device__ __forceinline__ void first_row(const RowsV<ST> &v, uint32_t a, int l, Acc &acc, unsigned *err,
                                          TupleShared &sh) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if constexpr (R == 2) {
        pairs_of<ST>(v, a, l, acc, err);
    } else {
        const uint32_t off = TU_OFF_LIST + (uint32_t)warp * TU_LIST_W;
        const uint32_t lt = (1u << lane) - 1u;
        uint32_t A[4];
#pragma unroll
        for (int w = 0; w < 4; w++) A[w] = w < (int)v.W ? v.word(w, a) : 0u;
        const uint32_t pa = row_positions<ST>(v, a, A);
        const uint32_t Wp = (pa + 31) / 32;
        bool fits = Wp <= 4 || R == 3;
        uint32_t m = 0;
        for (uint32_t cb = a + 1; fits && cb < v.n; cb += 32) {
            const uint32_t bal = survivors<ST>(v, a, A, cb, l, acc);
            if ((m + __popc(bal) + 3) * Wp > TU_LIST_W) {
                fits = false;
                break;
            }
            if ((bal >> lane) & 1u) sm_dyn[off + m + __popc(bal & lt)] = cb + lane;
            m += __popc(bal);
        }
        if (!fits) {
            // (row_units leaves room for every warp's entry)
            if (lane == 0) sh.defer[atomicAdd(&sh.ndefer, 1u)] = a;
            __syncwarp();
            return;
        }
        if (m < (uint32_t)(R - 1)) return;
        if (R > 3 && m >= CTA_LIST) {
            if (lane == 0) sh.defer[atomicAdd(&sh.ndefer, 1u)] = a;
            __syncwarp();
            return;
        }
        const uint32_t ms = (m + 3) & ~3u;
        __syncwarp();
        for (uint32_t kb = 0; kb < m; kb += 32) {
            const uint32_t k = kb + lane;
            const uint32_t c = sm_dyn[off + (k < m ? k : kb)];
            __syncwarp();
            project_row<ST>(v, a, c, off, m, ms, k);
        }
        __syncwarp();
        list_all<R>(off, m, ms, Wp, pa, 0, 1, l, acc, err);
        __syncwarp();
    }
}

// One first row on the whole CTA: its list takes the area of all warps' lists.
template <int R, bool ST>
__device__ void first_row_cta(const RowsV<ST> &v, uint32_t a, int l, Acc &acc, unsigned *err,
                              TupleShared &sh, uint32_t *scratch, uint32_t wmax) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t lt = (1u << lane) - 1u;
    __syncthreads();
    if (tid == 0) sh.m = 0;
    __syncthreads();
    uint32_t A[4];
#pragma unroll
    for (int w = 0; w < 4; w++) A[w] = w < (int)v.W ? v.word(w, a) : 0u;
    const uint32_t pa = row_positions<ST>(v, a, A);
    const uint32_t Wp = (pa + 31) / 32;
    bool fits = Wp <= 4 || R == 3;
    if (fits) {
        for (uint32_t cb = a + 1 + 32u * warp; cb < v.n; cb += 32u * TU_WARPS) {
            const uint32_t bal = survivors<ST>(v, a, A, cb, l, acc);
            uint32_t base = 0;
            if (lane == 0 && bal) base = atomicAdd(&sh.m, (unsigned)__popc(bal));
            base = __shfl_sync(FULL, base, 0);
            if (((bal >> lane) & 1u) && base + __popc(bal & lt) < TU_LISTS_W)
                sm_dyn[TU_OFF_LIST + base + __popc(bal & lt)] = cb + lane;
        }
        __syncthreads();
    }
    const uint32_t m = sh.m;
    const uint32_t ms = (m + 3) & ~3u;
    fits = fits && (unsigned long long)ms * Wp <= TU_LISTS_W;
    if (fits) {
        if (m < (uint32_t)(R - 1)) return;
        const uint32_t nb = (m + 31) / 32;
        if (v.W > 4 && nb <= TU_WARPS / 2) {
            // few rows of many words: the warps share the words too
            const uint32_t segs = TU_WARPS / nb, blk = (uint32_t)warp % nb, seg = (uint32_t)warp / nb;
            const uint32_t k = 32 * blk + lane;
            const uint32_t c = sm_dyn[TU_OFF_LIST + (k < m ? k : 32 * blk)];
            __syncthreads();
            for (uint32_t t = tid; t < ms * Wp; t += TU_THREADS) sm_dyn[TU_OFF_LIST + t] = 0;
            __syncthreads();
            if (seg < segs)
                project_words<ST>(v, a, c, v.W * seg / segs, v.W * (seg + 1) / segs, TU_OFF_LIST, m, ms, k);
        } else {
            // entry k of the index list is overwritten by its own first word only
            for (uint32_t kb = 32u * warp; kb < m; kb += 32u * TU_WARPS) {
                const uint32_t k = kb + lane;
                const uint32_t c = sm_dyn[TU_OFF_LIST + (k < m ? k : kb)];
                __syncwarp();
                project_row<ST>(v, a, c, TU_OFF_LIST, m, ms, k);
            }
        }
        __syncthreads();
        list_all<R>(TU_OFF_LIST, m, ms, Wp, pa, (uint32_t)warp, TU_WARPS, l, acc, err);
    } else {
        // masks of every level in the warp's list area, else in global scratch
        const bool in_sm = (unsigned long long)(R - 1) * v.W <= TU_LIST_W;
        uint32_t *scr = in_sm ? sm_dyn + TU_OFF_LIST + (uint32_t)warp * TU_LIST_W : scratch;
        const uint32_t ws = in_sm ? v.W : wmax;
        __syncthreads();
        for (uint32_t w = lane; w < v.W; w += 32) scr[w] = v.word(w, a);
        __syncwarp();
        for (uint32_t cb = a + 1 + 32u * warp; cb < v.n; cb += 32u * TU_WARPS)
            expand_wide<2, R, ST>(v, scr, ws, cb, cb + 32 < v.n ? cb + 32 : v.n, l, acc, err);
    }
}

// First rows of an anchor, claimed in batches by the warps (and by the
// anchor's other items when claim is set); with `wide` (see row_item) one at a
// time by the CTA.
template <int R, bool ST>
__device__ void row_units(const RowsV<ST> &v, uint32_t n_first, unsigned *claim, bool wide, int l, Acc &acc,
                          unsigned *err, TupleShared &sh, uint32_t *scratch, uint32_t wmax) {
    const int lane = threadIdx.x & 31;
    constexpr unsigned BATCH_MAX = R == 2 ? 4 : 1;
    const unsigned BATCH = v.W <= 8 ? BATCH_MAX : 1u;  // (a wide first row is work enough)
    for (;;) {
        // a round ends when the deferred rows could no longer be recorded
        __syncthreads();
        if (threadIdx.x == 0) {
            sh.ndefer = 0;
            if (R == 3 && wide) {
                const unsigned u = atomicAdd(claim, 1u);
                sh.defer[0] = u;
                sh.ndefer = u < n_first;
            }
        }
        __syncthreads();
        bool more = R == 3 && wide && sh.ndefer != 0;
        while (R != 3 || !wide) {
            if constexpr (R > 2) {
                // other warps add to the counter meanwhile: one lane reads it, so
                // that the warp leaves the loop together
                unsigned nd = 0;
                if (lane == 0) nd = *(volatile unsigned *)&sh.ndefer;
                nd = __shfl_sync(FULL, nd, 0);
                if (nd > DEFER_MAX - TU_WARPS * BATCH_MAX) {
                    more = true;
                    break;
                }
            }
            unsigned u = 0;
            if (lane == 0) u = atomicAdd(claim, BATCH);
            u = __shfl_sync(FULL, u, 0);
            if (u >= n_first) break;
            const unsigned ue = u + BATCH < n_first ? u + BATCH : n_first;
            for (; u < ue; u++) first_row<R, ST>(v, u, l, acc, err, sh);
        }
        if constexpr (R > 2) {
            more = __syncthreads_or(more);
            const unsigned nd = sh.ndefer;
            for (unsigned k = 0; k < nd; k++)
                first_row_cta<R, ST>(v, sh.defer[k], l, acc, err, sh, scratch, wmax);
        }
        if (!more) break;
    }
    __syncthreads();
}

// Row item: order the rows by ascending popcount (the same order in every item
// of the anchor), stage them, take first rows.
template <int R>
__device__ void row_item(const TupleArgs &a, const Item &it, Acc &acc, unsigned *err, TupleShared &sh,
                         uint32_t *scratch) {
    const int tid = threadIdx.x, lane = tid & 31;
    const uint32_t r = it.anchor, n = a.nrow[r], W = (a.dprime[r] + 31) / 32, stride = a.rsv_c[r];
    const uint32_t *region = a.pool + a.pool_off[r];
    const int l = a.l;
    unsigned *claim = it.claim == NO_CLAIM ? &sh.unit : a.claims + it.claim;
    uint16_t *perm = (uint16_t *)(sm_dyn + TU_OFF_PERM);
    const bool ordered = R > 2 && n <= TU_PERM;  // (the order of pairs does not matter)
    const uint32_t n_first = n - (uint32_t)R + 1;
    if (tid == 0) {
        sh.unit = 0;
        sh.n_units = it.claim == NO_CLAIM ? 0u : *(volatile unsigned *)claim;
        sh.words = 0;
    }
    bool wide = false;
    if (ordered) {
        for (int i = tid; i < 256; i += TU_THREADS) sh.hist[i] = 0;
        __syncthreads();
        if (sh.n_units >= n_first) return;  // the anchor's other items took everything
        uint16_t *key = (uint16_t *)(sm_dyn + TU_OFF_LIST);
        uint32_t words = 0;  // of the rows, each projected on itself
        for (uint32_t i = tid; i < n; i += TU_THREADS) {
            uint32_t p = 0;
            for (uint32_t w = 0; w < W; w++) p += __popc(region[(size_t)w * stride + i]);
            words += (p + 31) / 32;
            const uint32_t k = p < 255u ? p : 255u;
            key[i] = (uint16_t)k;
            atomicAdd(&sh.hist[k], 1u);
        }
        if (R == 3 && W > 4) {
            words = __reduce_add_sync(FULL, words);
            if (lane == 0) atomicAdd(&sh.words, words);
        }
        __syncthreads();
        // Three partners: where a typical first row with a quarter of the rows exceeds
        // a warp's list, nearly every first row goes to the CTA. Warps would defer
        // them as fast as they claim them, all to the first CTA that comes, and
        // the anchor's other items would find none left; the CTA takes them one at a
        // time. Tuples of four in 60 hubs of 500,000: 48 -> 8.8 ms, (4,2) of
        // K_{40,9000} 12.4 -> 4.0 (with the words of a projection shared by the
        // warps). More partners keep the warps: (5,5) of the 20k-edge graph took
        // 0.75 ms this way against 0.62, short lists being a warp's work there.
        if (R == 3 && W > 4) {
            const uint32_t wl = sh.words / n;  // of a typical list entry
            wide = R == 3 && wl > 4 && (n / 4 + 3) * wl > TU_LIST_W;
        }
        if (tid < 32) {
            uint32_t carry = 0;
            for (int b = 0; b < 256; b += 32) {  // exclusive scan of the bins
                const uint32_t x = sh.hist[b + lane];
                uint32_t s = x;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t t = __shfl_up_sync(FULL, s, o);
                    if (lane >= o) s += t;
                }
                sh.hist[b + lane] = carry + s - x;
                carry += __shfl_sync(FULL, s, 31);
            }
            __syncwarp();
            // stable placement, 32 rows at a time
            for (uint32_t b = 0; b < n; b += 32) {
                const uint32_t i = b + lane;
                const uint32_t k = i < n ? key[i] : 512u + lane;
                const uint32_t peers = __match_any_sync(FULL, k);
                const uint32_t rank = __popc(peers & ((1u << lane) - 1u));
                if (i < n) perm[sh.hist[k] + rank] = (uint16_t)i;
                __syncwarp();
                if (i < n && rank == 0) sh.hist[k] += __popc(peers);
                __syncwarp();
            }
        }
        __syncthreads();
    } else {
        __syncthreads();
        if (sh.n_units >= n_first) return;
    }
    if ((unsigned long long)n * W <= TU_ROWS_W) {
        for (uint32_t w = 0; w < W; w++)
            for (uint32_t i = tid; i < n; i += TU_THREADS)
                sm_dyn[w * n + i] = region[(size_t)w * stride + (ordered ? (uint32_t)perm[i] : i)];
        __syncthreads();
        RowsV<true> v;
        v.g = nullptr;
        v.perm = nullptr;
        v.stride = n;
        v.W = W;
        v.n = n;
        row_units<R, true>(v, n_first, claim, wide, l, acc, err, sh, scratch, a.wmax);
    } else {
        RowsV<false> v;
        v.g = region;
        v.perm = ordered ? perm : nullptr;
        v.stride = stride;
        v.W = W;
        v.n = n;
        row_units<R, false>(v, n_first, claim, wide, l, acc, err, sh, scratch, a.wmax);
    }
}

// ---- column walk: masks CM[q] of the rows that hold position q (wc row
// words at an odd stride wcp, so that lanes reading different columns hit
// different banks). A warp walks the position subsets depth first; at every
// node its lanes test 32 children at once, each intersecting the node's prefix
// (held one word per lane and broadcast by shuffles) with its column.

// A node's prefix mask, word w at lane w % 32, slot w / 32 (passed by value so
// that it stays in registers across calls).
template <int WPL>
struct Pfx {
    uint32_t m[WPL];
};

// Partial result of a subtree of the walk.
struct ColOut {
    U128 sum;
    uint32_t tested = 0, leaves = 0;
};

// Bound by a shuffle and a load per mask word and warp, four warps per scheduler:
// several words are in flight, and leaves read their binomial from a table. (One
// word at a time and 64-bit divisions: (4,4) of a dense 300 x 2000 graph with tuples
// from the 2000 868 ms, now 700; (3,4) 38, now 28; (4,5) of 400 x 400 88, now 72.)
// Children q in [qs, qe] of a node at depth LEV - 1 with prefix M; lanes over
// q. At depth l a child is a leaf and adds binom(N_Q, R); otherwise children
// with N >= R are expanded one at a time.
template <int R, int WPL, int LEV>
__device__ __noinline__ ColOut col_scan(uint32_t dp, uint32_t wc, uint32_t wcp, Pfx<WPL> M, uint32_t qs,
                                        uint32_t qe, int l, unsigned *err) {
    const int lane = threadIdx.x & 31;
    ColOut out;
    for (uint32_t qb = qs; qb <= qe; qb += 32) {
        const uint32_t q = qb + lane;
        const bool valid = q <= qe;
        const uint32_t o = (valid ? q : qs) * wcp;
        uint32_t n = 0;
#pragma unroll
        for (int k = 0; k < WPL; k++) {
            if (32u * k >= wc) break;  // WPL = 4 also serves 65..96 words
            const uint32_t wend = wc - 32u * k < 32u ? wc - 32u * k : 32u;
            // eight words at a time, then four, so that their loads and shuffles
            // overlap (words past the last meet a prefix of zeros)
            auto words = [&](uint32_t sl, auto blk) {
                constexpr int N = decltype(blk)::value;
                uint32_t x[N];
#pragma unroll
                for (int j = 0; j < N; j++) x[j] = sm_dyn[o + 32u * k + sl + j];
#pragma unroll
                for (int j = 0; j < N; j++) x[j] &= __shfl_sync(FULL, M.m[k], sl + j);
#pragma unroll
                for (int j = 0; j < N; j++) n += __popc(x[j]);
            };
            uint32_t sl = 0;
            for (; sl + 8 <= wend; sl += 8) words(sl, std::integral_constant<int, 8>());
            for (; sl < wend; sl += 4) words(sl, std::integral_constant<int, 4>());
        }
        out.tested += valid;
        if (LEV == l) {
            if (valid && n >= (uint32_t)R) {
                out.leaves++;
                if (n <= (uint32_t)BINOM_TBL) out.sum.add(s_btR[n]);
                else binom_add_k<R>(out.sum, n, err);
            }
        } else if constexpr (LEV < 8) {
            const uint32_t qe2 = dp - 1 - (uint32_t)(l - LEV - 1);  // room for the rest of Q
            uint32_t bal = __ballot_sync(FULL, valid && n >= (uint32_t)R);
            while (bal) {
                const uint32_t qc = qb + __ffs(bal) - 1;
                bal &= bal - 1;
                if (qc + 1 > qe2) continue;
                Pfx<WPL> X;
#pragma unroll
                for (int k = 0; k < WPL; k++) {
                    const uint32_t w = lane + 32u * k;
                    X.m[k] = w < wc ? (M.m[k] & sm_dyn[qc * wcp + w]) : 0u;
                }
                const ColOut c = col_scan<R, WPL, LEV + 1>(dp, wc, wcp, X, qc + 1, qe2, l, err);
                if (out.sum.add(c.sum)) atomicOr(err, CERR_OVERFLOW);
                out.tested += c.tested;
                out.leaves += c.leaves;
            }
        }
    }
    return out;
}

// A unit: first position q1 and a chunk of 32 second positions.
template <int R, int WPL>
__device__ void col_unit(uint32_t dp, uint32_t wc, uint32_t wcp, uint32_t q1, uint32_t chunk, int l,
                         Acc &acc, unsigned *err) {
    const int lane = threadIdx.x & 31;
    Pfx<WPL> M;
    uint32_t n = 0;
#pragma unroll
    for (int k = 0; k < WPL; k++) {
        const uint32_t w = lane + 32u * k;
        M.m[k] = w < wc ? sm_dyn[q1 * wcp + w] : 0u;
        n += __popc(M.m[k]);
    }
    n = __reduce_add_sync(FULL, n);
    if (n < (uint32_t)R) return;  // no Q through q1 has R rows
    const uint32_t qe2 = dp - 1 - (uint32_t)(l - 2);
    const uint32_t qs = q1 + 1 + 32u * chunk;
    if (qs > qe2) return;
    const uint32_t qe = qs + 31 < qe2 ? qs + 31 : qe2;
    const ColOut o = col_scan<R, WPL, 2>(dp, wc, wcp, M, qs, qe, l, err);
    if (acc.sum.add(o.sum)) atomicOr(err, CERR_OVERFLOW);
    acc.tested += o.tested;
    acc.leaves += o.leaves;
    acc.words += (unsigned long long)wc * o.tested;
}

template <int R>
__device__ void col_item(const TupleArgs &a, const Item &it, Acc &acc, unsigned *err, TupleShared &sh) {
    const int tid = threadIdx.x, lane = tid & 31;
    const uint32_t r = it.anchor, n = a.nrow[r], dp = a.dprime[r], W = (dp + 31) / 32, stride = a.rsv_c[r];
    const uint32_t *region = a.pool + a.pool_off[r];
    const int l = a.l;
    const uint32_t wc = (n + 31) / 32, wcp = wc | 1u;
    unsigned *claim = it.claim == NO_CLAIM ? &sh.unit : a.claims + it.claim;
    const uint32_t firsts = dp - (uint32_t)l + 1;
    const uint32_t chunks = (dp + 1 - (uint32_t)l + 31) / 32;  // of second positions, at most
    if (tid == 0) {
        sh.unit = 0;
        sh.n_units = it.claim == NO_CLAIM ? 0u : *(volatile unsigned *)claim;
    }
    __syncthreads();
    if (sh.n_units >= firsts * chunks) return;  // the anchor's other items took everything
    for (uint32_t t = tid; t < dp * wcp; t += TU_THREADS) sm_dyn[t] = 0;
    __syncthreads();
    for (uint32_t i = tid; i < n; i += TU_THREADS) {
        const uint32_t bit = 1u << (i & 31), cw = i >> 5;
        for (uint32_t w = 0; w < W; w++) {
            uint32_t x = region[(size_t)w * stride + i];
            while (x) {
                const int b = __ffs(x) - 1;
                x &= x - 1;
                atomicOr(&sm_dyn[(32 * w + b) * wcp + cw], bit);
            }
        }
    }
    __syncthreads();
    for (;;) {
        uint32_t u = 0;
        if (lane == 0) u = atomicAdd(claim, 1u);
        u = __shfl_sync(FULL, u, 0);
        if (u >= firsts * chunks) break;
        const uint32_t q1 = u / chunks, chunk = u - q1 * chunks;
        if (wc <= 32) col_unit<R, 1>(dp, wc, wcp, q1, chunk, l, acc, err);
        else if (wc <= 64) col_unit<R, 2>(dp, wc, wcp, q1, chunk, l, acc, err);
        else col_unit<R, 4>(dp, wc, wcp, q1, chunk, l, acc, err);
    }
    __syncthreads();
}

// ---- small anchors: one per warp, rows staged in the warp's list area
template <int R, int WN>
__device__ __forceinline__ void warp_rows(uint32_t off, uint32_t n, uint32_t W, uint32_t buf, int l,
                                          Acc &acc) {
    PrefixBuf<WN> pb;
    pb.off = off;
    pb.m = pb.ms = n;
    pb.W = W;
    pb.buf = buf;
    if constexpr (R == 2) {
        for (uint32_t b = 0; b < n; b += 32) {
            const uint32_t c = b + (threadIdx.x & 31);
            uint32_t T[WN];
#pragma unroll
            for (int w = 0; w < WN; w++) T[w] = c < n && w < (int)W ? sm_dyn[off + w * n + c] : 0u;
            pb.push(c + 1 < n, T, c, l, acc);
        }
    } else {
        for (uint32_t i = 0; i + (R - 1) < n; i++) {
            uint32_t pre[WN];
#pragma unroll
            for (int w = 0; w < WN; w++) pre[w] = w < (int)W ? sm_dyn[off + w * n + i] : 0u;
            expand<2, R, WN>(pb, pre, i + 1, l, acc);
        }
    }
    pb.flush(l, acc);
}

template <int R>
__device__ void warp_anchor(const TupleArgs &a, uint32_t r, Acc &acc, unsigned *err) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t off = TU_OFF_LIST + (uint32_t)warp * TU_LIST_W;
    const uint32_t n = a.nrow[r], W = (a.dprime[r] + 31) / 32, stride = a.rsv_c[r];
    const uint32_t *region = a.pool + a.pool_off[r];
    const int l = a.l;
    __syncwarp();
    for (uint32_t w = 0; w < W; w++)
        for (uint32_t i = lane; i < n; i += 32) sm_dyn[off + w * n + i] = region[(size_t)w * stride + i];
    __syncwarp();
    const uint32_t buf = TU_OFF_BUF + (uint32_t)warp * TU_BUF_W;
    if (W == 1) warp_rows<R, 1>(off, n, W, buf, l, acc);
    else if (W == 2) warp_rows<R, 2>(off, n, W, buf, l, acc);
    else warp_rows<R, 4>(off, n, W, buf, l, acc);
}

template <int R>
__global__ void __launch_bounds__(TU_THREADS, 1) k_tuples(const __grid_constant__ TupleArgs a) {
    __shared__ TupleShared sh;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    unsigned *err = &a.cnt->err;
    for (int x = tid; x <= BINOM_TBL; x += TU_THREADS) {
        unsigned long long v = 0;
        if (x >= a.l) {
            v = 1;
            for (int i = 1; i <= a.l; i++) v = v * (unsigned long long)(x - a.l + i) / (unsigned long long)i;
        }
        s_bt[x] = v;
        unsigned long long vr = 0;
        if (x >= R) {
            vr = 1;
            for (int i = 1; i <= R; i++) vr = vr * (unsigned long long)(x - R + i) / (unsigned long long)i;
        }
        s_btR[x] = vr;
        if (x <= TBL32) s_bt32[x] = (x >= a.l ? LEAF : 0u) | (uint32_t)(v & (LEAF - 1));
    }
    __syncthreads();
    if (tid == 0) {
        uint32_t x = 0;
        while (x < (uint32_t)TBL32 && s_bt[x + 1] < LEAF / 8) x++;
        s_max32 = x;
    }
    __syncthreads();
    uint32_t *scratch = a.wide_scratch
        ? a.wide_scratch + ((size_t)blockIdx.x * TU_WARPS + warp) * SCRATCH_SLOTS * a.wmax : nullptr;
    const unsigned n_items = a.cnt->n_items, n_warp = a.cnt->n_warp;
    const bool split_totals = a.tot.per_anchor || a.tot.per_graph;
    Acc acc;
    auto flush = [&](uint32_t r) {
        const U128 ws = warp_sum_u128(acc.sum, err);
        if (lane == 0) add_totals(a.tot, r, ws);
        acc.sum = U128();
    };
    for (;;) {
        __syncthreads();
        if (tid == 0) sh.item = atomicAdd(&a.cnt->head_b, 1u);
        __syncthreads();
        const unsigned item = sh.item;
        if (item >= n_items) break;
        const Item it = a.items[item];
        if (it.cols) col_item<R>(a, it, acc, err, sh);
        else row_item<R>(a, it, acc, err, sh, scratch);
        if (split_totals) flush(it.anchor);
    }
    // small anchors, one per warp
    while (n_warp) {
        unsigned k = 0;
        if (lane == 0) k = atomicAdd(&a.cnt->head_w, 1u);
        k = __shfl_sync(FULL, k, 0);
        if (k >= n_warp) break;
        const uint32_t r = a.warp_list[k];
        warp_anchor<R>(a, r, acc, err);
        if (split_totals) flush(r);
    }
    if (!split_totals) flush(0);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        acc.tested += __shfl_xor_sync(FULL, acc.tested, o);
        acc.leaves += __shfl_xor_sync(FULL, acc.leaves, o);
        acc.words += __shfl_xor_sync(FULL, acc.words, o);
    }
    if (lane == 0 && acc.tested) {
        atomicAdd(&a.cnt->tested, acc.tested);
        atomicAdd(&a.cnt->leaves, acc.leaves);
        atomicAdd(&a.cnt->popc_words, acc.words);
    }
}
