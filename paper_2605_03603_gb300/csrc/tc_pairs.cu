// Tensor-core form of the two-partner tuple step (Algorithm 2, Section 4.3,
// the loop over (p-1)-subsets A of C with p - 1 = 2, and the type count of
// Section 4.2) for anchors whose candidate masks are wide.
//
// An anchor's rows are the parts S_c = P_c AND NOT D_c (common neighbours where
// sign(u,v) = sign(c,v)) and T_c = P_c AND D_c (where they differ) of its
// candidates that hold at least l positions, as 0/1 vectors over its useful
// positions. For a pair of candidates i < j the four type classes of Section
// 4.2 are (s,s), (s,d), (d,s), (d,d), with sizes <S_i,S_j>, <S_i,T_j>,
// <T_i,S_j>, <T_i,T_j>; the two parts of one candidate are disjoint (product 0,
// which adds nothing). With Z the rows stacked, the anchor therefore adds, over
// row pairs a < b, binom(G[a][b], l) with G = Z Z^T. This is a dense
// contraction over the positions, so it runs on the tensor cores:
//
// * k_zexpand writes Z as fp8 e4m3 bytes in 16 KB blocks of 128 rows x 128
//   positions, each block already in the shared-memory layout of the MMA
//   (K-major, 128-byte swizzle: 16-byte chunk c of row r at chunk c ^ (r & 7)),
//   so a block moves to shared memory with one plain bulk copy. A set bit is
//   the byte 0x08 = 2^-6, so a product is 2^-12 and every sum an exact multiple
//   of it.
// * k_tcpairs is a persistent kernel over output tiles of 128 x 256 rows of G
//   (only tiles that hold a pair a < b). Per CTA one thread issues the bulk
//   copies and one tcgen05.mma (kind::f8f6f4, M = 128, N = 256, K = 32 per
//   instruction; 512 cycles per 128 positions) into one of two TMEM
//   accumulators; the fp32 accumulator holds the sums exactly (at most d' <
//   2^21 < 2^24 units of 2^-12). The tiles of a column of 256 rows follow one
//   another, so their B blocks stay in shared memory for the run (anchors of at
//   most 384 positions) and a tile reads only its A block, 16 KB instead of
//   48 KB per 128 positions. (Expanding the bits in the kernel instead, four
//   warps per block, was slower: 1,325 cycles per block.)
//   Sixteen epilogue warps read the accumulator with tcgen05.ld and add
//   binom(G[a][b], l): the sum of l! binom(x, l) = x (x - 1) .. (x - l + 1) in
//   packed fp32 multiply-adds, exact below 2^24, 1 to 2 instructions per entry
//   and no shared-memory lookups; long rows take a table (32-bit, or 64-bit
//   with exact 128-bit arithmetic above 256). The packed chains are bound by
//   latency, hence four warps per scheduler.
//   Work comes in jobs of consecutive tiles of one anchor, whose records every
//   role prefetches one ahead; the loops of the copying and the issuing thread
//   run over the blocks of a run of tiles (their instructions, a few cycles
//   each, were 2,100 cycles per tile when every tile was set up anew), and a
//   chunk's anchors share one epilogue, so each kernel holds only its own.
//
// Every wait on an mbarrier is bounded by a clock limit; a wait that runs out
// sets the error word, every role stops, copies and MMAs in flight are waited
// for (again bounded), TMEM is freed and the kernel returns.
#include <algorithm>
#include <vector>

#include "sbc_internal.cuh"

namespace sbc {

namespace {

constexpr int TC_EPI_WARPS = 16;   // warps 2..17: four per TMEM lane group, 64 columns each
constexpr int TC_THREADS = 32 * (2 + TC_EPI_WARPS);  // warp 0 MMA, warp 1 copies
constexpr uint32_t TC_BLOCK = 16384;           // one operand block: 128 rows x 128 bytes
constexpr int TC_A = 7;                        // ring of A blocks (128 rows)
constexpr int TC_B = 3;                        // ring of B block pairs (256 rows)
constexpr size_t TC_SMEM = (size_t)(TC_A + 2 * TC_B) * TC_BLOCK + 1024;  // + alignment slack
constexpr int TC_TMEM_COLS = 512;              // two 128 x 256 fp32 accumulators
constexpr int TC_BINOM = 256;
constexpr long long TC_WAIT_CYCLES = 4000000000ll;  // about 2 s at the SM clock

// kind::f8f6f4 instruction descriptor: D f32, A and B e4m3, both K-major,
// N = 256, M = 128.
constexpr uint32_t TC_IDESC = (1u << 4) | (0u << 7) | (0u << 10) | ((256u >> 3) << 17) |
                              ((128u >> 4) << 24);

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count)
                 : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
                 "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint64_t *bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Bounded wait for the phase of parity `parity` to complete. Returns false
// when the CTA aborts (this wait ran out, or another role's did).
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, volatile int *abort_flag,
                                          unsigned *err) {
    if (mbar_try(bar, parity)) return true;
    const long long t0 = clock64();
    for (;;) {
        // try_wait suspends the thread in hardware until the phase completes
        // or a short time limit passes, so this loop needs no sleep of its own
        if (mbar_try(bar, parity)) return true;
        if (*abort_flag) return false;
        if (clock64() - t0 > TC_WAIT_CYCLES) {
            *abort_flag = 1;
            atomicOr(err, kErrTimeout);
            return false;
        }
    }
}

// One bulk copy of `bytes` (a multiple of 16, both addresses 16-byte
// aligned) from global to shared memory, completing on `bar`.
__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, uint32_t bytes, uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
            "r"(smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}

// Shared-memory matrix descriptor (K-major, 128-byte swizzle, 8-row groups 1024
// bytes apart): the upper word is the stride byte offset, the version and the
// swizzle mode, the lower word the address in 16-byte units and the (unused)
// leading byte offset. Four MMAs cover a 128-position block, 32 bytes each.
constexpr uint32_t TC_DESC_HI = (1024u >> 4) | (1u << 14) | (2u << 29);
__device__ __forceinline__ uint32_t desc_lo(uint32_t saddr) { return (saddr >> 4) | (1u << 16); }

__device__ __forceinline__ void tc_mma(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t accum) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
        "setp.ne.b32 p, %5, 0;\n\t"
        "mov.b64 da, {%1, %3};\n\t"
        "mov.b64 db, {%2, %3};\n\t"
        "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], da, db, %4, p;\n\t}" ::"r"(d_tmem),
        "r"(a_lo), "r"(b_lo), "r"(TC_DESC_HI), "r"(TC_IDESC), "r"(accum));
}
__device__ __forceinline__ void tc_commit(uint64_t *bar) {
    asm volatile(
        "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
            smem_u32(bar))
        : "memory");
}
__device__ __forceinline__ void tc_fence_before() {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// 32 consecutive fp32 columns of this thread's TMEM lane: the load is issued,
// and its registers may be read after tmem_wait on them.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&v)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
          "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]),
          "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]), "=r"(v[17]), "=r"(v[18]),
          "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]),
          "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]),
          "=r"(v[31])
        : "r"(taddr));
}
// Waits for every load this warp issued; the operands keep uses of v after it.
__device__ __forceinline__ void tmem_wait(uint32_t (&v)[32]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]),
                   "+r"(v[7]), "+r"(v[8]), "+r"(v[9]), "+r"(v[10]), "+r"(v[11]), "+r"(v[12]),
                   "+r"(v[13]), "+r"(v[14]), "+r"(v[15]), "+r"(v[16]), "+r"(v[17]), "+r"(v[18]),
                   "+r"(v[19]), "+r"(v[20]), "+r"(v[21]), "+r"(v[22]), "+r"(v[23]), "+r"(v[24]),
                   "+r"(v[25]), "+r"(v[26]), "+r"(v[27]), "+r"(v[28]), "+r"(v[29]), "+r"(v[30]),
                   "+r"(v[31])
                 :
                 : "memory");
}

// Packed pairs of fp32 (two lanes of one 64-bit register).
__device__ __forceinline__ uint64_t f2_pack(uint32_t a, uint32_t b) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(a), "r"(b));
    return r;
}
__device__ __forceinline__ void f2_unpack(uint64_t v, uint32_t &a, uint32_t &b) {
    asm("mov.b64 {%0, %1}, %2;" : "=r"(a), "=r"(b) : "l"(v));
}
__device__ __forceinline__ uint64_t f2_add(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t f2_mul(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t f2_fma(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ uint64_t f2_both(float x) {
    return f2_pack(__float_as_uint(x), __float_as_uint(x));
}

// Longest row up to which the packed epilogue is exact. FLOAT: 16 values of
// x (x - 1) .. (x - l + 1) per fp32 lane sum below 2^24. INT: one value stays
// below 2^23, so that value + 2^23 carries it in its low bits; 128 of them sum
// below 2^32.
template <int L, bool INT>
__host__ __device__ constexpr uint32_t tc_poly_max() {
    if (L < 2 || L > 4) return 0;
    uint32_t best = 0;
    for (uint32_t x = L; x <= 2048; x++) {
        unsigned long long f = 1;
        for (int i = 0; i < L; i++) f *= x - i;
        if (INT ? f >= (1ull << 23) : 16 * f >= (1ull << 24)) break;
        best = x;
    }
    return best;
}

// Accumulator entries are multiples of this unit; 2^23 units as a float.
constexpr float TC_UNIT = 1.0f / 4096.0f;
constexpr uint32_t TC_BASE = 0x4B000000u - (12u << 23);

// Sum of x (x - 1) .. (x - L + 1) over the 32 entries (integers in units of
// TC_UNIT, so the product carries TC_UNIT^L); with MASK only over the entries
// j >= first.
template <int L, bool INT, bool MASK>
__device__ __forceinline__ uint32_t poly_sum(const uint32_t (&v)[32], int first) {
    uint64_t acc = f2_both(0.0f);
    constexpr float U = TC_UNIT, UL = L == 2 ? U * U : L == 3 ? U * U * U : U * U * U * U;
    const uint64_t base = f2_both(8388608.0f * UL), m1 = f2_both(-U), m3 = f2_both(-3.0f * U),
                   p2 = f2_both(2.0f * U * U);
    uint32_t isum = 0;
#pragma unroll
    for (int j = 0; j < 32; j += 2) {
        uint64_t x;
        if constexpr (MASK) x = f2_pack(j >= first ? v[j] : 0u, j + 1 >= first ? v[j + 1] : 0u);
        else x = f2_pack(v[j], v[j + 1]);
        // the last factor is multiplied into the accumulator
        uint64_t a, b;
        if constexpr (L == 2) {
            a = x;
            b = f2_add(x, m1);
        } else if constexpr (L == 3) {
            a = f2_fma(x, f2_add(x, m3), p2);
            b = x;
        } else {
            a = f2_mul(x, f2_add(x, m3));
            b = f2_add(a, p2);
        }
        if constexpr (INT) {
            uint32_t r0, r1;
            f2_unpack(f2_fma(a, b, base), r0, r1);
            isum += r0 + r1;
        } else {
            acc = f2_fma(a, b, acc);
        }
    }
    if constexpr (INT) {
        // a power of two times the integer: only the exponent field differs
        constexpr uint32_t EXP = 0x4B000000u - (12u * L << 23);
        return isum - 32u * EXP;
    }
    uint32_t r0, r1;
    f2_unpack(acc, r0, r1);
    return (uint32_t)(__uint_as_float(r0) * (1.0f / UL)) + (uint32_t)(__uint_as_float(r1) * (1.0f / UL));
}

// binom(x, l) exactly for x > TC_BINOM (128-bit multiplicative formula; the
// running value after step i is binom(x - l + i, i), so dividing before
// multiplying by the reduced factor keeps it exact). Sets kErrOverflow when
// the value needs more than 128 bits.
__device__ __noinline__ U128 tc_binom_big(unsigned long long x, int l, unsigned *err) {
    unsigned long long lo = 1, hi = 0;
    for (int i = 1; i <= l; i++) {
        unsigned long long f = x - l + i;
        unsigned long long g = (unsigned long long)i, h = f % g;  // g = gcd(f, i)
        while (h) {
            const unsigned long long t = g % h;
            g = h;
            h = t;
        }
        // divide (hi, lo) by i / g (exact: it divides the running value)
        const unsigned long long dv = (unsigned long long)i / g;
        if (dv > 1) {
            unsigned long long qh = hi / dv, rem = hi % dv;
            unsigned long long a = (rem << 32) | (lo >> 32);
            unsigned long long q1 = a / dv;
            rem = a % dv;
            unsigned long long b = (rem << 32) | (lo & 0xFFFFFFFFull);
            hi = qh;
            lo = (q1 << 32) | (b / dv);
        }
        const unsigned long long m = f / g;
        unsigned long long l0 = lo * m, c = __umul64hi(lo, m);
        unsigned long long h0 = hi * m, hh = __umul64hi(hi, m);
        unsigned long long nh = h0 + c;
        if (hh != 0 || nh < h0) {
            atomicOr(err, kErrOverflow);
            return U128();
        }
        lo = l0;
        hi = nh;
    }
    U128 t;
    t.lo = lo;
    t.hi = hi;
    return t;
}

}  // namespace

// Expand the chunk's rows into Z blocks (see the file comment). A CTA expands
// consecutive blocks: one search for its first anchor, then a walk over the few
// anchors of its range (with strided blocks every CTA walked the records of all
// anchors, a dependent load each). Eight lanes write one row's 128 bytes, so a
// warp's store covers four whole lines (one row per lane wrote a sixteenth of
// 32 lines at a time).
__global__ void __launch_bounds__(512) k_zexpand(TcArgs a) {
    const int64_t per = (a.n_blocks + gridDim.x - 1) / gridDim.x;
    const int64_t b0 = blockIdx.x * per, b1 = b0 + per < a.n_blocks ? b0 + per : a.n_blocks;
    if (b0 >= b1) return;
    int ai = 0, hi = a.n_anc;  // largest ai with zblk0 <= b0
    while (hi - ai > 1) {
        const int mid = (ai + hi) >> 1;
        if (a.anc[mid].zblk0 <= b0) ai = mid; else hi = mid;
    }
    TcAnchor A = a.anc[ai];
    const uint32_t c = threadIdx.x & 7;  // 16-byte chunk: positions 16 c .. 16 c + 15
    uint32_t rb = (uint32_t)((b0 - A.zblk0) / A.KB), kb = (uint32_t)((b0 - A.zblk0) % A.KB);
    for (int64_t blk = b0; blk < b1; blk++) {
        const uint32_t w = 4 * kb + (c >> 1);
#pragma unroll
        for (int h = 0; h < 2; h++) {
            const uint32_t r = (threadIdx.x >> 3) + 64 * h, row = rb * 128 + r;
            uint32_t bits = 0;
            if (row < A.nr && w < A.W) bits = a.pool[A.pool_off + (int64_t)w * A.rsv + row] >> ((c & 1) * 16);
            // each nibble is spread to bit 3 of 4 bytes
            uint32_t o[4];
#pragma unroll
            for (int k = 0; k < 4; k++) o[k] = (((bits >> (4 * k)) & 0xFu) * 0x01020408u) & 0x08080808u;
            *reinterpret_cast<uint4 *>(a.z + blk * (int64_t)TC_BLOCK + r * 128 + ((c ^ (r & 7)) << 4)) =
                make_uint4(o[0], o[1], o[2], o[3]);
        }
        if (++kb == A.KB) {
            kb = 0;
            if (++rb == A.RB && blk + 1 < b1) {
                rb = 0;
                A = a.anc[++ai];
            }
        }
    }
}

namespace {

// Jobs of every anchor (thread per anchor).
__global__ void k_tcjobs(const TcAnchor *anc, int n_anc, int job_tiles, TcJob *jobs) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n_anc; i += gridDim.x * blockDim.x) {
        const TcAnchor A = anc[i];
        TcJob j;
        j.zblk0 = A.zblk0;
        j.r = A.r;
        j.KB = A.KB;
        j.longest = A.longest;
        for (uint32_t t = 0; t < A.tiles; t += job_tiles) {
            j.local = t;
            j.count = A.tiles - t < (uint32_t)job_tiles ? A.tiles - t : (uint32_t)job_tiles;
            jobs[A.job0 + t / job_tiles] = j;
        }
    }
}

// Walks the runs of one CTA: jobs blockIdx.x, + gridDim.x, ..., each some
// consecutive tiles of one anchor. Block coordinates of a tile: I rows of 128,
// J columns of 256; column J holds the rows I = 0 .. 2J + 1 (the tiles with a
// pair a < b), so J (J + 1) tiles come before it. A run is the tiles of a job in
// one column: rows I .. I + n - 1. The next job's record is loaded while this
// one runs.
struct RunCursor {
    TcJob A, ahead;
    int64_t job;       // of `ahead`
    uint32_t left = 0; // tiles of this job after the current run
    uint32_t I = 0, J = 0, n = 0;
    __device__ __forceinline__ RunCursor(const TcArgs &a) : job(blockIdx.x) {
        if (job < a.n_jobs) ahead = a.jobs[job];
    }
    __device__ __forceinline__ bool next(const TcArgs &a) {
        if (left) {
            I = 0;
            J++;
        } else {
            if (job >= a.n_jobs) return false;
            A = ahead;
            job += gridDim.x;
            if (job < a.n_jobs) ahead = a.jobs[job];
            left = A.count;
            J = (uint32_t)((sqrtf(4.0f * (float)A.local + 1.0f) - 1.0f) * 0.5f);
            while (J * (J + 1) > A.local) J--;
            while ((J + 1) * (J + 2) <= A.local) J++;
            I = A.local - J * (J + 1);
        }
        n = min(left, 2 * J + 2 - I);
        left -= n;
        return true;
    }
};

}  // namespace

// binom(x, L) in 64 bits by the multiplicative formula (every partial
// product fits when x <= the host's 64-bit limit for L); the divisors are
// compile-time constants.
template <int L>
__device__ __forceinline__ unsigned long long binom_u64c(unsigned long long x) {
    unsigned long long r = 1;
#pragma unroll
    for (int i = 1; i <= L; i++) r = r * (x - L + i) / (unsigned long long)i;
    return r;
}

// Largest multiple of 32 (at most 2048) with 32 * binom(x, L) < 2^32: for
// anchors whose longest row has at most this many positions every Gram entry
// indexes a 32-bit table and 32 of its binomials sum in 32 bits.
template <int L>
__host__ __device__ constexpr uint32_t tc_fast_max() {
    uint32_t best = 0;
    for (uint32_t x = 32; x <= 2048; x += 32) {
        unsigned long long b = 1;
        for (int i = 1; i <= L; i++) b = b * (x - L + i) / i;
        if (32ull * b >= (1ull << 32)) break;
        best = x;
    }
    return best;
}

// Epilogue of a chunk's anchors, by their longest row: packed fp32 sums, packed
// with integer sums, tables.
enum : int { EPI_FLOAT = 0, EPI_INT = 1, EPI_TABLE = 2 };

template <int L, int EPI>
__global__ void __launch_bounds__(TC_THREADS, 1) k_tcpairs(const __grid_constant__ TcArgs a) {
    extern __shared__ __align__(16) unsigned char tc_smem_raw[];
    __shared__ __align__(8) uint64_t full_a[TC_A], empty_a[TC_A], full_b[TC_B], empty_b[TC_B];
    __shared__ __align__(8) uint64_t acc_full[2], acc_empty[2], mma_done;
    __shared__ uint32_t s_tmem;
    __shared__ volatile int s_abort;
    // binom(x, L) for x <= TC_BINOM, zero below L and at TC_BINOM + 1 (the
    // clamped index of larger entries, which a slower path adds), and for x <=
    // FAST in 32 bits (anchors whose longest row is that short)
    constexpr uint32_t FAST = tc_fast_max<L>();
    __shared__ unsigned long long s_bt[EPI == EPI_TABLE ? TC_BINOM + 2 : 1];
    __shared__ uint32_t s_bt32[EPI == EPI_TABLE ? FAST + 1 : 1];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    unsigned char *smem =
        (unsigned char *)(((uintptr_t)tc_smem_raw + 1023) & ~(uintptr_t)1023);
    if constexpr (EPI == EPI_TABLE) {
        for (int x = tid; x <= TC_BINOM + 1; x += TC_THREADS)
            s_bt[x] = (x >= L && x <= TC_BINOM) ? binom_u64c<L>(x) : 0ull;
        for (int x = tid; x <= (int)FAST; x += TC_THREADS)
            s_bt32[x] = x >= L ? (uint32_t)binom_u64c<L>(x) : 0u;
    }
    if (tid == 0) {
        for (int s = 0; s < TC_A; s++) {
            mbar_init(&full_a[s], 1);
            mbar_init(&empty_a[s], 1);
        }
        for (int s = 0; s < TC_B; s++) {
            mbar_init(&full_b[s], 1);
            mbar_init(&empty_b[s], 1);
        }
        for (int b = 0; b < 2; b++) {
            mbar_init(&acc_full[b], 1);
            mbar_init(&acc_empty[b], TC_EPI_WARPS);
        }
        mbar_init(&mma_done, 1);
        s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(&s_tmem)),
                     "r"(TC_TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;
    unsigned char *smem_b = smem + (size_t)TC_A * TC_BLOCK;

    if (warp == 1) {
        // ---- copies. A run's A blocks are consecutive in Z. With KB <= TC_B the
        // run's B pairs come first and stay; else pair kb before A block kb.
        if (lane == 0) {
            uint32_t sa = 0, ra = 0, sb = 0, rb = 0;  // ring slots and rounds
            uint32_t used_a = 0, used_b = 0;          // slots ever filled
            RunCursor tr(a);
            auto push_a = [&](const unsigned char *z) -> bool {
                if (!mbar_wait(&empty_a[sa], (ra & 1) ^ 1, &s_abort, a.err)) return false;
                mbar_expect_tx(&full_a[sa], TC_BLOCK);
                bulk_g2s(smem + (size_t)sa * TC_BLOCK, z, TC_BLOCK, &full_a[sa]);
                used_a |= 1u << sa;
                if (++sa == TC_A) {
                    sa = 0;
                    ra++;
                }
                return true;
            };
            auto push_b = [&](const unsigned char *z0, const unsigned char *z1) -> bool {
                if (!mbar_wait(&empty_b[sb], (rb & 1) ^ 1, &s_abort, a.err)) return false;
                unsigned char *st = smem_b + (size_t)sb * 2 * TC_BLOCK;
                mbar_expect_tx(&full_b[sb], 2 * TC_BLOCK);
                bulk_g2s(st, z0, TC_BLOCK, &full_b[sb]);
                bulk_g2s(st + TC_BLOCK, z1, TC_BLOCK, &full_b[sb]);
                used_b |= 1u << sb;
                if (++sb == TC_B) {
                    sb = 0;
                    rb++;
                }
                return true;
            };
            bool ok = true;
            while (ok && !s_abort && tr.next(a)) {
                const uint32_t KB = tr.A.KB;
                const size_t row_bytes = (size_t)KB * TC_BLOCK;  // of one row of blocks
                const unsigned char *z = a.z + tr.A.zblk0 * (int64_t)TC_BLOCK;
                const unsigned char *zA = z + tr.I * row_bytes;
                const unsigned char *zB = z + 2 * tr.J * row_bytes;
                if (KB <= (uint32_t)TC_B) {
                    for (uint32_t kb = 0; kb < KB && ok; kb++)
                        ok = push_b(zB + kb * TC_BLOCK, zB + row_bytes + kb * TC_BLOCK);
                    const uint32_t blocks = tr.n * KB;
                    for (uint32_t b = 0; b < blocks && ok; b++, zA += TC_BLOCK) ok = push_a(zA);
                } else {
                    for (uint32_t i = 0; i < tr.n && ok; i++)
                        for (uint32_t kb = 0; kb < KB && ok; kb++, zA += TC_BLOCK)
                            ok = push_b(zB + (size_t)kb * TC_BLOCK, zB + row_bytes + (size_t)kb * TC_BLOCK) &&
                                 push_a(zA);
                }
            }
            if (s_abort) {
                // let every copy this thread started land before the CTA exits
                // (a slot's last round is one less where the ring has not
                // reached it again)
                for (int s = 0; s < TC_A; s++)
                    if ((used_a >> s) & 1u) {
                        const uint32_t last = (uint32_t)s < sa ? ra : ra - 1;
                        const long long t0 = clock64();
                        while (!mbar_try(&full_a[s], last & 1) && clock64() - t0 < TC_WAIT_CYCLES) {
                        }
                    }
                for (int s = 0; s < TC_B; s++)
                    if ((used_b >> s) & 1u) {
                        const uint32_t last = (uint32_t)s < sb ? rb : rb - 1;
                        const long long t0 = clock64();
                        while (!mbar_try(&full_b[s], last & 1) && clock64() - t0 < TC_WAIT_CYCLES) {
                        }
                    }
            }
        }
        __syncwarp();
    } else if (warp == 0) {
        // ---- MMA issue
        if (lane == 0) {
            uint32_t sa = 0, ra = 0, sb = 0, rb = 0, it = 0;
            const uint32_t alo = desc_lo(smem_u32(smem)), blo = desc_lo(smem_u32(smem_b));
            RunCursor tr(a);
            bool ok = true;
            // one 128-position step: A slot sa against the B pair at blk
            auto step = [&](uint32_t d_tmem, uint32_t pair, uint32_t accum) -> bool {
                if (!mbar_wait(&full_a[sa], ra & 1, &s_abort, a.err)) return false;
                tc_fence_after();
                const uint32_t pa = alo + sa * (TC_BLOCK >> 4), pb = blo + pair * (2 * TC_BLOCK >> 4);
                tc_mma(d_tmem, pa, pb, accum);
                tc_mma(d_tmem, pa + 2, pb + 2, 1);
                tc_mma(d_tmem, pa + 4, pb + 4, 1);
                tc_mma(d_tmem, pa + 6, pb + 6, 1);
                tc_commit(&empty_a[sa]);
                if (++sa == TC_A) {
                    sa = 0;
                    ra++;
                }
                return true;
            };
            while (ok && !s_abort && tr.next(a)) {
                const uint32_t KB = tr.A.KB;
                const bool resident = KB <= (uint32_t)TC_B;
                const uint32_t b0 = sb;  // the run's first pair
                for (uint32_t i = 0; i < tr.n && ok; i++, it++) {
                    const uint32_t buf = it & 1;
                    if (!mbar_wait(&acc_empty[buf], ((it >> 1) & 1) ^ 1, &s_abort, a.err)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    uint32_t pair = b0;
                    for (uint32_t kb = 0; kb < KB && ok; kb++) {
                        if (!resident || i == 0) {
                            pair = sb;
                            if (!mbar_wait(&full_b[sb], rb & 1, &s_abort, a.err)) {
                                ok = false;
                                break;
                            }
                            if (++sb == TC_B) {
                                sb = 0;
                                rb++;
                            }
                        }
                        ok = step(tmem + buf * 256, pair, kb != 0 ? 1u : 0u);
                        if (!resident) tc_commit(&empty_b[pair]);
                        if (++pair == TC_B) pair = 0;
                    }
                    if (ok) tc_commit(&acc_full[buf]);
                }
                if (resident && ok) {
                    // the run's pairs are free once its MMAs are done
                    uint32_t pair = b0;
                    for (uint32_t k = 0; k < KB; k++) {
                        tc_commit(&empty_b[pair]);
                        if (++pair == TC_B) pair = 0;
                    }
                }
            }
            // every MMA this thread issued has completed before TMEM is freed
            tc_commit(&mma_done);
            const long long t0 = clock64();
            while (!mbar_try(&mma_done, 0) && clock64() - t0 < TC_WAIT_CYCLES) {
            }
        }
        __syncwarp();
    } else {
        // ---- epilogue: warp w reads TMEM lanes 32 * (w % 4) .. (the rows of
        // its lane group) and 64 of the columns
        const uint32_t g = (uint32_t)(warp & 3);
        const uint32_t col0 = 64u * ((uint32_t)(warp - 2) >> 2);
        uint32_t it = 0;
        RunCursor tr(a);
        // the warp's sum over its tiles of one anchor, added to the totals
        // when the anchor changes (one set of atomics per anchor, not per tile)
        U128 sum;
        unsigned long long fsum = 0;  // the packed sums' L! binom(x, L)
        constexpr unsigned long long LFACT = L == 2 ? 2 : L == 3 ? 6 : 24;
        bool any = false, ok = true;
        uint32_t sum_r = 0;
        auto flush = [&]() {
            if constexpr (EPI != EPI_TABLE) {
                sum.add(fsum / LFACT);
                fsum = 0;
            }
            const U128 ws = warp_sum_u128(sum, a.err);
            if (lane == 0 && (ws.lo | ws.hi)) {
                atomic_add_u128(a.total, ws.lo, ws.hi, a.per_graph ? nullptr : a.err);
                if (a.per_anchor) atomic_add_u128(a.per_anchor + 2 * (size_t)sum_r, ws.lo, ws.hi, a.err);
                if (a.per_graph) {
                    int lo = 0, hi = a.n_graphs;  // largest graph with graph_x0 <= r
                    while (hi - lo > 1) {
                        const int mid = (lo + hi) >> 1;
                        if (a.graph_x0[mid] <= (int64_t)sum_r) lo = mid; else hi = mid;
                    }
                    atomic_add_u128(a.per_graph + 2 * (size_t)lo, ws.lo, ws.hi, a.err);
                }
            }
            sum = U128();
        };
        // binom(x, L) of entries above the table (rare: larger common sets)
        auto add_big = [&](uint32_t x) {
            if (x <= a.big64) sum.add(binom_u64c<L>(x));
            else if (sum.add(tc_binom_big(x, L, a.err))) atomicOr(a.err, kErrOverflow);
        };
        // 32 columns from column cb; kept: the columns >= c0 (per lane)
        auto chunk = [&](const uint32_t (&v)[32], uint32_t cb, uint32_t c0, bool fast) {
            const bool whole = cb >= c0;
            if constexpr (EPI != EPI_TABLE) {
                constexpr bool INT = EPI == EPI_INT;
                if (__all_sync(0xffffffffu, whole)) fsum += poly_sum<(L <= 4 ? L : 4), INT, false>(v, 0);
                else fsum += poly_sum<(L <= 4 ? L : 4), INT, true>(v, (int)c0 - (int)cb);
            } else if (fast) {
                // The float bits of entry + 2^23 units are TC_BASE + entry; the
                // table's address is offset by that constant (32-bit
                // shared-window arithmetic), and the bits are clamped to the
                // table's end. Dropped columns read entry 0.
                const uint32_t tb = smem_u32(s_bt32) - (TC_BASE << 2);
                uint32_t part32 = 0;
#pragma unroll
                for (int j = 0; j < 32; j++) {
                    const uint32_t x = whole || cb + j >= c0 ? v[j] : 0u;
                    const uint32_t bits =
                        min(__float_as_uint(__uint_as_float(x) + 8388608.0f * TC_UNIT), TC_BASE + FAST);
                    uint32_t b;
                    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(b) : "r"(tb + (bits << 2)));
                    part32 += b;
                }
                sum.add((unsigned long long)part32);
            } else {
                unsigned long long part = 0;  // < 32 * binom(256, 8) < 2^64
                uint32_t mx = 0;
#pragma unroll
                for (int j = 0; j < 32; j++) {
                    // the entry is an exact integer below 2^23 units: adding
                    // 2^23 of them leaves it in the low mantissa bits
                    uint32_t x = __float_as_uint(__uint_as_float(v[j]) + 8388608.0f * TC_UNIT) & 0x7FFFFFu;
                    x = cb + j >= c0 ? x : 0u;
                    mx = max(mx, x);
                    part += s_bt[min(x, (uint32_t)TC_BINOM + 1)];
                }
                sum.add(part);
                if (mx > (uint32_t)TC_BINOM) {
#pragma unroll
                    for (int j = 0; j < 32; j++) {
                        const uint32_t x =
                            __float_as_uint(__uint_as_float(v[j]) + 8388608.0f * TC_UNIT) & 0x7FFFFFu;
                        if (x > (uint32_t)TC_BINOM && cb + j >= c0) add_big(x);
                    }
                }
            }
        };
        while (ok && tr.next(a)) {
            if (!any || tr.A.r != sum_r) {
                if (any) flush();
                any = true;
                sum_r = tr.A.r;
            }
            const bool fast = tr.A.longest <= FAST;
            for (uint32_t i = 0; i < tr.n; i++, it++) {
                const uint32_t buf = it & 1;
                if (lane == 0) ok = mbar_wait(&acc_full[buf], (it >> 1) & 1, &s_abort, a.err);
                ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
                if (!ok) break;
                tc_fence_after();
                // columns of this tile (0..255) after the row: all of them off
                // the diagonal, from c0 on it
                const uint32_t row = (tr.I + i) * 128 + g * 32 + lane;  // row of G
                const uint32_t c0 = row + 1 > tr.J * 256 ? row + 1 - tr.J * 256 : 0u;
                const uint32_t cl0 = __shfl_sync(0xffffffffu, c0, 0);  // smallest in the warp
                // 32-column chunks from the first that holds a kept column of
                // some lane (warp-uniform)
                const uint32_t begin = max(col0, cl0 & ~31u), end = col0 + 64;
                const uint32_t tcol = tmem + ((g * 32) << 16) + buf * 256;
                uint32_t v[32];
                for (uint32_t cb = begin; cb < end; cb += 32) {
                    tmem_ld32(tcol + cb, v);
                    tmem_wait(v);
                    if (cb + 32 >= end) {
                        // the last chunk is in registers: the accumulator is
                        // free for the next tile but one
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&acc_empty[buf]);
                    }
                    chunk(v, cb, c0, fast);
                }
                if (begin >= end) {
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&acc_empty[buf]);
                }
            }
        }
        if (any) flush();
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "r"(TC_TMEM_COLS)
                     : "memory");
    }
}

namespace {

// Epilogue of an anchor whose longest row has x positions.
template <int L>
constexpr int epi_of(uint32_t x) {
    return x <= tc_poly_max<L, false>() ? EPI_FLOAT : x <= tc_poly_max<L, true>() ? EPI_INT : EPI_TABLE;
}
int epi_of(int l, uint32_t x) {
    return l == 2 ? epi_of<2>(x) : l == 3 ? epi_of<3>(x) : l == 4 ? epi_of<4>(x) : (int)EPI_TABLE;
}

const void *tc_kernel(int l, int epi) {
    switch (l) {
        case 2: return epi == EPI_FLOAT ? (const void *)k_tcpairs<2, EPI_FLOAT>
                     : epi == EPI_INT ? (const void *)k_tcpairs<2, EPI_INT> : (const void *)k_tcpairs<2, EPI_TABLE>;
        case 3: return epi == EPI_FLOAT ? (const void *)k_tcpairs<3, EPI_FLOAT>
                     : epi == EPI_INT ? (const void *)k_tcpairs<3, EPI_INT> : (const void *)k_tcpairs<3, EPI_TABLE>;
        case 4: return epi == EPI_FLOAT ? (const void *)k_tcpairs<4, EPI_FLOAT>
                     : epi == EPI_INT ? (const void *)k_tcpairs<4, EPI_INT> : (const void *)k_tcpairs<4, EPI_TABLE>;
        case 5: return (const void *)k_tcpairs<5, EPI_TABLE>;
        case 6: return (const void *)k_tcpairs<6, EPI_TABLE>;
        case 7: return (const void *)k_tcpairs<7, EPI_TABLE>;
        default: return (const void *)k_tcpairs<8, EPI_TABLE>;
    }
}

}  // namespace

// ------------------------------------------------------------------ host

TcPlan tc_plan(const std::vector<TcInput> &in, int l, int64_t budget_bytes) {
    TcPlan plan;
    std::vector<TcInput> v(in);
    // one epilogue per chunk; in it the heaviest per-tile work first, so that
    // the strided job assignment of the persistent kernel ends with short tiles
    std::sort(v.begin(), v.end(), [l](const TcInput &x, const TcInput &y) {
        const int ex = epi_of(l, x.longest), ey = epi_of(l, y.longest);
        return ex != ey ? ex > ey : x.W != y.W ? x.W > y.W : x.nr > y.nr;
    });
    TcChunk cur;
    auto flush = [&]() {
        if (cur.host.empty()) return;
        // up to 64 tiles amortise a job's start; fewer when that would not give
        // every SM several jobs
        cur.job_tiles = (int)std::max<int64_t>(1, std::min<int64_t>(64, cur.n_tiles / (152 * 16)));
        for (TcAnchor &A : cur.host) {
            A.job0 = cur.n_jobs;
            cur.n_jobs += ((int64_t)A.tiles + cur.job_tiles - 1) / cur.job_tiles;
        }
        plan.max_blocks = std::max(plan.max_blocks, cur.n_blocks);
        plan.tiles += cur.n_tiles;
        plan.chunks.push_back(std::move(cur));
        cur = TcChunk();
    };
    for (const TcInput &x : v) {
        TcAnchor A;
        A.r = x.r;
        A.nr = x.nr;
        A.W = x.W;
        A.rsv = x.rsv;
        A.longest = x.longest;
        A.pool_off = x.pool_off;
        const uint64_t h = (x.nr + 255) / 256;
        A.RB = (uint32_t)(2 * h);
        A.KB = (x.W + 3) / 4;
        // sum over columns J < h of 2J + 2, less the last tile when it has no rows
        const uint64_t tiles = h * (h + 1) - (((x.nr + 127) / 128) & 1);
        if (tiles > 0xFFFFFFFFull) fail(SBC_E_UNSUPPORTED, "an anchor with %u rows is too large", x.nr);
        A.tiles = (uint32_t)tiles;
        const int64_t nb = (int64_t)A.RB * A.KB;
        const int epi = epi_of(l, x.longest);
        if (!cur.host.empty() &&
            (epi != cur.epi || (cur.n_blocks + nb) * (int64_t)TC_BLOCK > budget_bytes)) flush();
        cur.epi = epi;
        A.zblk0 = cur.n_blocks;
        A.job0 = 0;
        cur.n_blocks += nb;
        cur.n_tiles += (int64_t)tiles;
        plan.kblocks += tiles * A.KB;
        cur.host.push_back(A);
        plan.anchors++;
    }
    flush();
    return plan;
}

void tc_upload(TcPlan &plan, cudaStream_t s) {
    for (TcChunk &c : plan.chunks) {
        c.dev.alloc(c.host.size(), s);
        SBC_CUDA(cudaMemcpyAsync(c.dev.ptr, c.host.data(), sizeof(TcAnchor) * c.host.size(),
                                 cudaMemcpyHostToDevice, s));
        c.jobs.alloc((size_t)c.n_jobs, s);
        k_tcjobs<<<grid_for((int64_t)c.host.size(), 128), 128, 0, s>>>(c.dev.ptr, (int)c.host.size(),
                                                                      c.job_tiles, c.jobs.ptr);
        SBC_LAUNCHED();
        g_launches++;
    }
}

void tc_ensure_attrs() {
    static std::mutex mu;
    static bool done[64] = {};
    std::lock_guard<std::mutex> lock(mu);
    int dev = 0;
    SBC_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) fail(SBC_E_UNSUPPORTED, "device ordinal %d out of range", dev);
    if (done[dev]) return;
    for (int l = 2; l <= 8; l++)
        for (int e = l <= 4 ? (int)EPI_FLOAT : (int)EPI_TABLE; e <= EPI_TABLE; e++)
            SBC_CUDA(cudaFuncSetAttribute(tc_kernel(l, e), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)TC_SMEM));
    done[dev] = true;
}

void tc_launch(const TcPlan &plan, TcArgs base, unsigned char *z, cudaStream_t s) {
    const int sms = sm_count();
    for (const TcChunk &c : plan.chunks) {
        TcArgs a = base;
        a.anc = c.dev.ptr;
        a.n_anc = (int)c.host.size();
        a.jobs = c.jobs.ptr;
        a.n_jobs = c.n_jobs;
        a.n_blocks = c.n_blocks;
        a.z = z;
        k_zexpand<<<(int)std::min<int64_t>(c.n_blocks, (int64_t)sms * 16), 512, 0, s>>>(a);
        SBC_LAUNCHED();
        const int g = (int)std::min<int64_t>(c.n_jobs, (int64_t)sms);
        void *args[] = {&a};
        SBC_CUDA(cudaLaunchKernel(tc_kernel(a.l, c.epi), dim3(g), dim3(TC_THREADS), args, TC_SMEM, s));
        SBC_LAUNCHED();
        g_launches += 2;
    }
}

}  // namespace sbc
