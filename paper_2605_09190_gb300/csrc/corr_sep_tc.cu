// corr_sep_tc.cu -- (a2) the separable exact correlation (sep.cuh) on the
// 5th-generation tensor cores, sides 64 and 128 (the latter: the DCT-II family
// alone, in the second half of the file): the same exact integer T = B Y B^T
// per family as the SIMT twin (corr_sep.cu), rounded the same way, so both
// give identical bits.
//
// At side 64 a CTA takes two leaves at a time: 128 rows of a tile are (leaf,
// row), and every value ends in the lane and the thread that uses it.
//
// Digits.  Bf = sum_{s<6} d_s 2^(8s) with balanced digits |d_s| <= 128 (the top
// one <= 45 in a DCT-II row of side 64, 181 in a Haar row), all exact BF16
// values, as are the centred pixels.  The bounds on their sums below are
// checked against the digits there are when the table is made (host.cu).
//   Fold (DCT-II).  Row q of Bf equals (-1)^q times its mirror image, so row m
//   of the pixels becomes y~[m] + y~[63-m] (m < 32) or y~[m] - y~[63-m]
//   (m >= 32), in place: at most 256 in magnitude, exact BF16.  The even rows
//   of Bf need the first 32 only, the odd ones the last 32: half of stage 2.
//   Stage 1: Z~^T[m][p] = sum_i y~[i][m] Bf[p][i].  A = the pixels (rows
//     (leaf, m), K = i), B = the digits (rows (parity of p, s, p / 2)): lane
//     (leaf, m) holds the six digit sums of each p, each at most 0.42 x 2^22
//     in magnitude: exact.  They are joined in int64 with the centring
//     term 128 R[p] of each pixel row (R[p] the row sums of Bf; a difference
//     has none) and split into eight balanced base-2^8 digits e_t, written to
//     shared memory as stage 2's A operand: rows (leaf, p), K = m, M-major, so
//     that a lane's row m is a row of 64 p there.
//   Stage 2: T[p][q] = sum_{t,s} 2^(8(t+s)) sum_m e_t[p][m] d_s[q][m], 32 q of
//     one parity at a time.  B = the digits d_0 .. d_5 of those q stacked (192
//     rows), so that one MMA with A = e_t adds into the columns of the digit
//     diagonals t .. t + 5 (32 columns each): the sum of at most six digit
//     products, 128 times a row's digits, at most 0.39 x 2^22: exact.  Without
//     the fold (the Haar family) K = 64, and 0.34 x 2^22 (a Haar row of 64
//     nonzero entries is a power of two, with one nonzero digit).
//   The epilogue joins the 13 diagonals of an output: adjacent ones in one
//   32-bit multiply-add on their biased bit patterns (no wrap), those as
//   disjoint words of two 128-bit numbers, and biased_to_df rounds the sum
//   plus one constant for all biases.
//
// What bounds it: the instructions of the epilogue and of the digit split
// (about 105 an output and 35 a value of Z~), which therefore overlap the MMAs where they can:
// a pass's outputs are rounded and stored while the next pass or the next
// pair's stage 1 runs.  Side 64, DCT-II family, 50 910 leaves: 5.26 -> 1.53
// ms (one leaf at a time with two digits in the 128 rows, halves that met
// through shared memory, 24 accumulators an output and the general rounding,
// before).
//
// One CTA per SM (16 warps, all 512 TMEM columns: stage 1 in 0..383, stage 2
// in 0..415), persistent over the pairs; thread 0 issues the TMA loads and the
// MMAs, all threads drain.  Every wait is bounded by a timer; on expiry the
// kernel waits, bounded again, for what it has in flight, records
// AQMP_E_TIMEOUT, frees its TMEM and returns.
#include <cuda.h>
#include <cuda_runtime.h>
#include <cuda_bf16.h>

#include "common.cuh"
#include "kernels.h"
#include "sep.cuh"
#include "tc_sep.cuh"

namespace aqmp {

namespace septc {

constexpr int kB = 64;                        // block side served here
constexpr int kThreads = 512;                 // 16 warps: 4 per TMEM lane quarter
constexpr int kTmemCols = 512;
constexpr int kTileY = 64 * 128;              // bytes: 64 rows (m) x 64 BF16 (i)
constexpr int kTileE = 64 * 128;              // bytes: 64 rows (m) x 64 BF16 (p) of one leaf and digit
constexpr int kDigitRows = 6 * 64;            // rows of one family: (parity, s, p / 2)
constexpr int kOffD = 0;
constexpr int kOffE = kOffD + kDigitRows * 128;          // [digit t][leaf]
constexpr int kOffY = kOffE + 8 * 2 * kTileE;            // [buffer][leaf]
constexpr int kOffCen = kOffY + 2 * 2 * kTileY;          // centring terms by p
constexpr int kOffBar = kOffCen + 8 * kB;                // barriers: digits, Y[2], MMA
constexpr int kOffMisc = kOffBar + 8 * 8;
constexpr int kSmemBytes = kOffMisc + 16 + 1024;

// M = 128, N columns; BF16 x BF16 -> F32; A K-major, or M-major in stage 2.
constexpr uint32_t idesc(int n, bool a_m_major) {
    return (1u << 4) | (1u << 7) | (1u << 10) | (a_m_major ? 1u << 15 : 0u) | ((uint32_t)(n >> 3) << 17) |
           ((uint32_t)(128 >> 4) << 24);
}

// M-major tile: rows k of 64 M values (128 bytes, 128-byte swizzle), groups of
// 8 k 1024 bytes apart; the second 64 M values one leaf's tile further.
__device__ __forceinline__ unsigned long long smem_desc_m_major(uint32_t addr) {
    unsigned long long d = 0;
    d |= (unsigned long long)((addr & 0x3ffffu) >> 4);
    d |= (unsigned long long)(kTileE >> 4) << 16;
    d |= (unsigned long long)(1024 >> 4) << 32;
    d |= (unsigned long long)1 << 46;
    d |= (unsigned long long)2 << 61;
    return d;
}

__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t (&r)[4]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(taddr));
}

__device__ __forceinline__ void fence_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// Two FP32 integers of magnitude below 2^22 as a 2^8 + b + kPairBias, without
// wrapping; one as a + kOneBias.
constexpr uint32_t kOneBias = 0x4B400000u, kPairBias = (uint32_t)(257ull * kOneBias);
__device__ __forceinline__ uint32_t biased_one(uint32_t bits) {
    return __float_as_uint(__fadd_rn(__uint_as_float(bits), 12582912.0f));
}
__device__ __forceinline__ uint32_t biased_pair(uint32_t a_bits, uint32_t b_bits) {
    return biased_one(a_bits) * 256u + biased_one(b_bits);
}

// Z~ + 128 in every byte from its six digit sums; c the centring term.
__device__ __forceinline__ unsigned long long join_digits(uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t a4,
                                                          uint32_t a5, unsigned long long c) {
    constexpr unsigned long long kC = 0x8080808080808080ull - (unsigned long long)kPairBias * 0x100010001ull;
    return (unsigned long long)biased_pair(a1, a0) + ((unsigned long long)biased_pair(a3, a2) << 16) +
           ((unsigned long long)biased_pair(a5, a4) << 32) + (kC + c);
}

// The words of T + the rounding's bias from output i's 13 diagonals.
__device__ __forceinline__ void join_diagonals(const uint32_t (&a)[13][4], int i, uint32_t (&T)[4]) {
    typedef unsigned __int128 u128;
    constexpr u128 kPairs = (u128)kPairBias * ((((u128)1 << 48 | (u128)1 << 32) | ((u128)1 << 16 | 1)) |
                                               ((u128)1 << 80 | (u128)1 << 64));
    constexpr u128 kC = (((u128)kDigitBiasHi << 64) | kDigitBiasLo) - kPairs - ((u128)kOneBias << 96);
    const u128 even = (u128)biased_pair(a[1][i], a[0][i]) | (u128)biased_pair(a[5][i], a[4][i]) << 32 |
                      (u128)biased_pair(a[9][i], a[8][i]) << 64 | (u128)biased_one(a[12][i]) << 96;
    const u128 odd = (u128)biased_pair(a[3][i], a[2][i]) << 16 | (u128)biased_pair(a[7][i], a[6][i]) << 48 |
                     (u128)biased_pair(a[11][i], a[10][i]) << 80;
    const u128 t = even + odd + kC;
    T[0] = (uint32_t)t;
    T[1] = (uint32_t)(t >> 32);
    T[2] = (uint32_t)(t >> 64);
    T[3] = (uint32_t)(t >> 96);
}

// The 13 diagonals of 8 columns from column `col` of each 32, joined.
__device__ __forceinline__ void drain_diagonals(uint32_t lane_base, int col, uint32_t (&T)[8][4]) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        uint32_t a[13][4];
#pragma unroll
        for (int c = 0; c < 13; ++c) tmem_ld4(lane_base + 32 * c + col + 4 * h, a[c]);
        wait_ld();
#pragma unroll
        for (int i = 0; i < 4; ++i) join_diagonals(a, i, T[4 * h + i]);
    }
}

// x + y and y - x of two 16-byte chunks of BF16, in place.
__device__ __forceinline__ void fold_chunks(uint4 *pa, uint4 *pb) {
    uint4 x = *pa, y = *pb;
    auto both = [](uint32_t &u, uint32_t &v) {
        uint32_t s, d;
        asm("add.rn.bf16x2 %0, %1, %2;" : "=r"(s) : "r"(u), "r"(v));
        asm("sub.rn.bf16x2 %0, %1, %2;" : "=r"(d) : "r"(v), "r"(u));
        u = s;
        v = d;
    };
    both(x.x, y.x);
    both(x.y, y.y);
    both(x.z, y.z);
    both(x.w, y.w);
    *pa = x;
    *pb = y;
}

// Stage 2's MMAs over the 16-wide steps k0 .. k1: every digit tile of E
// against the six stacked digits at D (192 rows), into the diagonals' columns.
__device__ __forceinline__ void issue_stage2(uint32_t tmem, uint32_t sE, uint32_t sD, int k0, int k1) {
    for (int kk = k0; kk < k1; ++kk) {
        const uint32_t more = kk > k0 ? 1u : 0u;
        const unsigned long long ad = smem_desc_m_major(sE) + 128ull * kk;
        const unsigned long long bd = smem_desc(sD) + 2ull * kk;
        constexpr unsigned long long kStepE = 2 * kTileE >> 4;
        // digits 0 and 6 meet every diagonal but the last first
        mma_ss(tmem, ad, bd, idesc(192, true), more);
        mma_ss(tmem + 192, ad + 6 * kStepE, bd, idesc(192, true), more);
        mma_ss(tmem + 224, ad + 7 * kStepE, bd, idesc(160, true), 1u);
        mma_ss(tmem + 384, ad + 7 * kStepE, bd + (5 * 32 * 128 >> 4), idesc(32, true), more);
        for (int t = 1; t < 6; ++t) mma_ss(tmem + 32 * t, ad + t * kStepE, bd, idesc(192, true), 1u);
    }
}

}  // namespace septc

// Y map: the gathered leaves viewed as [capacity * 64 rows][64] BF16 (row m of
// leaf l at row 64 l + m, K = i); digit map: [2 * 384 rows][64] BF16, the rows
// of family F from 384 F.
__global__ void __launch_bounds__(septc::kThreads, 1)
corr_sep_tc_kernel(const __grid_constant__ CUtensorMap tmY, const __grid_constant__ CUtensorMap tmD, int F, int M,
                   int off, const long long *__restrict__ Rs, const unsigned *count_dev, long long fixed_count,
                   float2 *__restrict__ c0, Counters *ctr) {
    using namespace septc;
    const long long count = count_dev ? (long long)*count_dev : fixed_count;
    const long long pairs = (count + 1) / 2;
    if ((long long)blockIdx.x >= pairs) return;                  // uniform
    const bool fold = F == 0;

    extern __shared__ unsigned char smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    unsigned char *gbase = smem_raw + (base - raw);
    const uint32_t sD = base + kOffD, sE = base + kOffE, sY = base + kOffY, sBar = base + kOffBar;
    const uint32_t barD = sBar, barY0 = sBar + 8, barY1 = sBar + 16, barMma = sBar + 24;
    unsigned long long *cen = reinterpret_cast<unsigned long long *>(gbase + kOffCen);
    uint32_t *tmem_holder = reinterpret_cast<uint32_t *>(gbase + kOffMisc);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        mbar_init(barD, 1);
        mbar_init(barY0, 1);
        mbar_init(barY1, 1);
        mbar_init(barMma, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(tmem_holder)), "r"(kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    // the centring of Z~'s rows: 128 R[p], twice that for a sum of two rows
    if (tid < kB) cen[tid] = (unsigned long long)(Rs[F * kB + tid] * (fold ? 256 : 128));
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = *tmem_holder;

    auto load_pair = [&](long long pair, int buf) {
        const uint32_t bar = buf ? barY1 : barY0;
        mbar_expect_tx(bar, 2 * kTileY);
        for (int l = 0; l < 2; ++l)                              // a row past the end reads zeros
            tma_load_2d(sY + (2 * buf + l) * kTileY, &tmY, bar, 0, (int)(64 * (2 * pair + l)));
    };
    // the digits once, the first pair's pixels
    if (tid == 0) {
        mbar_expect_tx(barD, kDigitRows * 128);
        for (int t = 0; t < 3; ++t) tma_load_2d(sD + t * 128 * 128, &tmD, barD, 0, kDigitRows * F + 128 * t);
        load_pair(blockIdx.x, 0);
    }
    bool ok = __syncthreads_and(mbar_wait(barD, 0)) != 0;

    // TMEM lane quarter of this warp and the column group it drains
    const int quarter = warp & 3, cg = warp >> 2;
    const int row = quarter * 32 + lane, half = row >> 6, r64 = row & 63;      // (leaf, m) or (leaf, p)
    const uint32_t lane_base = tmem + ((uint32_t)(quarter * 32) << 16);
    const bool difference = fold && (quarter & 1);                             // rows m >= 32
    uint32_t mma_phase = 0, y_phase[2] = {0u, 0u};
    uint32_t T[8][4];                                                          // biased words, 8 q of a pass

    // rounds and stores the outputs q = 2 (8 cg + j) + par of a pair
    auto finish = [&](long long pair, int par) {
        const long long leaf = 2 * pair + half;
        if (leaf >= count) return;
        float2 *out = c0 + leaf * M + off + (2 * 8 * cg + par) * kB + r64;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const df v = biased_to_df(T[j][0], T[j][1], T[j][2], T[j][3]);
            out[2 * j * kB] = make_float2(v.hi, v.lo);
        }
    };

    int it = 0;
    long long pending = -1;
    for (long long pair = blockIdx.x; ok && pair < pairs; pair += gridDim.x, ++it) {
        const int buf = it & 1;
        ok = __syncthreads_and(mbar_wait(buf ? barY1 : barY0, y_phase[buf])) != 0;
        if (!ok) break;
        y_phase[buf] ^= 1u;
        // prefetch the next pair into the other buffer (its last reader, the
        // previous pair's stage 1, has been waited for)
        if (tid == 0 && pair + gridDim.x < pairs) load_pair(pair + gridDim.x, buf ^ 1);
        if (fold) {
            // rows m and 63 - m, one 16-byte chunk a thread (the swizzle places
            // chunk j of row m at j ^ (m mod 8))
            const int l = tid >> 8, m = (tid >> 3) & 31, j = tid & 7;
            unsigned char *t = gbase + kOffY + (2 * buf + l) * kTileY;
            uint4 *pa = reinterpret_cast<uint4 *>(t + m * 128 + ((j ^ (m & 7)) << 4));
            uint4 *pb = reinterpret_cast<uint4 *>(t + (63 - m) * 128 + ((j ^ (7 - (m & 7))) << 4));
            fold_chunks(pa, pb);
            fence_async();
        }
        fence_before();
        __syncthreads();
        // ---- stage 1
        if (tid == 0) {
            fence_after();
            const unsigned long long ad = smem_desc(sY + 2 * buf * kTileY), bd = smem_desc(sD);
#pragma unroll
            for (int par = 0; par < 2; ++par)
#pragma unroll
                for (int kk = 0; kk < 4; ++kk)
                    mma_ss(tmem + 192 * par, ad + 2ull * kk, bd + (unsigned long long)(par * 192 * 128 >> 4) + 2ull * kk,
                           idesc(192, false), kk > 0 ? 1u : 0u);
            mma_commit(barMma);
        }
        if (pending >= 0) finish(pending, 1);
        ok = __syncthreads_and(mbar_wait(barMma, mma_phase)) != 0;
        if (!ok) break;
        mma_phase ^= 1u;
        fence_after();
        // ---- drain 1: p = 16 cg + 8 h + (0 .. 7), one chunk of each digit's row
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            uint32_t a[2][6][4];
#pragma unroll
            for (int par = 0; par < 2; ++par)
#pragma unroll
                for (int sd = 0; sd < 6; ++sd) tmem_ld4(lane_base + 192 * par + 32 * sd + 8 * cg + 4 * h, a[par][sd]);
            wait_ld();
            uint32_t e[8][4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                uint32_t lo[2], hi[2];
#pragma unroll
                for (int par = 0; par < 2; ++par) {
                    const unsigned long long z =
                        join_digits(a[par][0][i], a[par][1][i], a[par][2][i], a[par][3][i], a[par][4][i], a[par][5][i],
                                    difference ? 0ull : cen[16 * cg + 8 * h + 2 * i + par]);
                    lo[par] = (uint32_t)z;
                    hi[par] = (uint32_t)(z >> 32);
                }
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    e[t][i] = bytes_less_128(lo[0], lo[1], t);
                    e[4 + t][i] = bytes_less_128(hi[0], hi[1], t);
                }
            }
            unsigned char *dst = gbase + kOffE + half * kTileE + r64 * 128 + (((2 * cg + h) ^ (r64 & 7)) << 4);
#pragma unroll
            for (int t = 0; t < 8; ++t)
                *reinterpret_cast<uint4 *>(dst + t * 2 * kTileE) = make_uint4(e[t][0], e[t][1], e[t][2], e[t][3]);
        }
        fence_async();
        fence_before();
        __syncthreads();
        // ---- stage 2, the q of one parity a pass
#pragma unroll 1
        for (int par = 0; par < 2 && ok; ++par) {
            if (tid == 0) {
                fence_after();
                issue_stage2(tmem, sE, sD + par * 192 * 128, fold ? 2 * par : 0, fold ? 2 * par + 2 : 4);
                mma_commit(barMma);
            }
            if (par == 1) finish(pair, 0);
            ok = __syncthreads_and(mbar_wait(barMma, mma_phase)) != 0;
            if (!ok) break;
            mma_phase ^= 1u;
            fence_after();
            // ---- drain 2: q = 2 (8 cg + j) + par, 13 diagonals each
            drain_diagonals(lane_base, 8 * cg, T);
            fence_before();
            __syncthreads();
        }
        pending = pair;
    }
    if (ok && pending >= 0) finish(pending, 1);
    if (tid == 0 && !ok) {
        // what may be in flight, before shared memory and TMEM are given up: the
        // phase that each barrier is at
        mbar_wait(barD, 0);
        mbar_wait(barY0, y_phase[0]);
        mbar_wait(barY1, y_phase[1]);
        mbar_wait(barMma, mma_phase);
    }
    fence_before();
    __syncthreads();
    if (tid == 0 && !ok && ctr) raise_error(ctr, kDevErrTimeout, 12u);
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
}

// ------------------------------------------------------------- side 128
//
// The DCT-II family, one leaf at a time: the 128 rows of stage 1's tile are the
// folded pixel rows m (64 sums, 64 differences), K = i = 128, and the digit
// sums stay below 128 x 256 x 128 = 2^22 (the top digit is at most 32).  The
// digits e_t of one class of rows (128 p, K = 64 m) fill 128 KB, so the classes
// b = 0, 1 (the even and the odd q) go one after the other, and stage 1's
// products are formed for one parity a of p at a time (384 columns), of which a
// class's half of the rows is drained.  Stage 2 as at side 64, 32 of the class's
// q a pass; its digit sums reach 0.99 x 2^22 for the rows there are (checked
// when the table is made).
//   The six digits of all 128 rows take 192 KB: they come through one 48 KB
// buffer, as (parity of the row, half of K) chunks.  Class b takes (1 - b, 1 - b)
// first, which the class before left there, then (1 - b, b), (b, 1 - b) and
// (b, b), which is also stage 2's operand.
//   A 17th warp loads and issues, so that the 16 that drain round and store a
// pass's outputs meanwhile.  M is ordered (p / 16, a, p' mod 8), p' = p / 2, so
// that a thread writes whole chunks and a warp's 32 outputs are contiguous.
// 3072 leaves: 0.62 ms; both families of the SIMT twin took 3.65 ms, bound by
// the wide integer multiply-adds, and the Haar family alone takes 0.24.
namespace septc {
constexpr int kThreads128 = 17 * 32;
constexpr int kChunk = 384 * 128;                                // bytes of a digit chunk
constexpr int kOffE128 = 0;
constexpr int kOffD128 = kOffE128 + 8 * 2 * kTileE;
constexpr int kOffY128 = kOffD128 + kChunk;                      // [half of K][128 rows]
constexpr int kOffCen128 = kOffY128 + 2 * 128 * 128;
constexpr int kOffBar128 = kOffCen128 + 8 * 128;                 // digits, pixels, producer's, drainers', back
constexpr int kOffMisc128 = kOffBar128 + 8 * 8;
constexpr int kSmemBytes128 = kOffMisc128 + 16 + 1024;
}  // namespace septc

// Y map: [capacity * 128 rows][128] BF16 in boxes of 128 rows x 64; digit map:
// [2 * 768 rows][128] BF16, row (a, q half, s, q mod 32 of the parity) of a family.
__global__ void __launch_bounds__(septc::kThreads128, 1)
corr_sep_tc128_kernel(const __grid_constant__ CUtensorMap tmY, const __grid_constant__ CUtensorMap tmD, int M,
                      const long long *__restrict__ Rs, const unsigned *count_dev, long long fixed_count,
                      float2 *__restrict__ c0, Counters *ctr) {
    using namespace septc;
    constexpr int b = 128;
    const long long count = count_dev ? (long long)*count_dev : fixed_count;
    if ((long long)blockIdx.x >= count) return;                  // uniform

    extern __shared__ unsigned char smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    unsigned char *gbase = smem_raw + (base - raw);
    const uint32_t sE = base + kOffE128, sD = base + kOffD128, sY = base + kOffY128, sBar = base + kOffBar128;
    const uint32_t barD = sBar, barY = sBar + 8, barP = sBar + 16, barA = sBar + 24, barC = sBar + 32;
    unsigned long long *cen = reinterpret_cast<unsigned long long *>(gbase + kOffCen128);
    uint32_t *tmem_holder = reinterpret_cast<uint32_t *>(gbase + kOffMisc128);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        mbar_init(barD, 1);
        mbar_init(barY, 1);
        mbar_init(barP, 1);
        mbar_init(barA, 1);
        mbar_init(barC, 16);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(tmem_holder)), "r"(kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid < b) cen[tid] = (unsigned long long)(Rs[tid] * 256);      // of a sum of two rows
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = *tmem_holder;
    bool ok = true;

    if (warp == 16) {
        if (lane == 0) {
            uint32_t phD = 0, phP = 0, phC = 0;
            uint32_t nD = 0, nY = 0, nP = 0, nA = 0;              // issued on each barrier
            auto load_digits = [&](int a, int kh) {
                ++nD;
                mbar_expect_tx(barD, kChunk);
                for (int t = 0; t < 3; ++t) tma_load_2d(sD + t * 128 * 128, &tmD, barD, 64 * kh, 384 * a + 128 * t);
            };
            auto load_pixels = [&](long long leaf) {
                ++nY;
                mbar_expect_tx(barY, 2 * 128 * 128);
                for (int kh = 0; kh < 2; ++kh) tma_load_2d(sY + kh * 128 * 128, &tmY, barY, 64 * kh, (int)(128 * leaf));
            };
            auto wait = [&](uint32_t bar, uint32_t &phase) {
                ok = ok && mbar_wait(bar, phase);
                phase ^= 1u;
                return ok;
            };
            // stage 1 over one half of K
            auto stage1 = [&](int kh, uint32_t acc, uint32_t bar) {
                fence_after();
                const unsigned long long ad = smem_desc(sY + kh * 128 * 128), bd = smem_desc(sD);
                for (int qh = 0; qh < 2; ++qh)
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk)
                        mma_ss(tmem + 192 * qh, ad + 2ull * kk, bd + (unsigned long long)(qh * 192 * 128 >> 4) + 2ull * kk,
                               idesc(192, false), kk > 0 ? 1u : acc);
                mma_commit(bar);
                ++(bar == barP ? nP : nA);
            };
            load_digits(1, 1);
            load_pixels(blockIdx.x);
            bool fresh = true;
            for (long long leaf = blockIdx.x; ok && leaf < count; leaf += gridDim.x) {
                for (int cls = 0; cls < 2 && ok; ++cls) {
                    if (!wait(barC, phC)) break;                  // pixels folded, accumulators drained
                    if (fresh && !wait(barD, phD)) break;
                    fresh = false;
                    stage1(1 - cls, 0u, barP);                    // chunk (1 - cls, 1 - cls)
                    if (!wait(barP, phP)) break;
                    load_digits(1 - cls, cls);
                    if (!wait(barD, phD)) break;
                    stage1(cls, 1u, barA);
                    ok = mbar_wait(barA, 0);                      // four completions a class: parities 0, 1, 0, 1
                    if (!ok) break;
                    load_digits(cls, 1 - cls);
                    if (!wait(barC, phC) || !wait(barD, phD)) break;
                    stage1(1 - cls, 0u, barP);
                    if (!wait(barP, phP)) break;
                    load_digits(cls, cls);
                    if (!wait(barD, phD)) break;
                    stage1(cls, 1u, barA);
                    ok = mbar_wait(barA, 1);
                    if (!ok) break;
                    if (cls == 1 && leaf + gridDim.x < count) load_pixels(leaf + gridDim.x);
                    for (int qh = 0; qh < 2 && ok; ++qh) {
                        if (!wait(barC, phC)) break;              // digits written; the pass before drained
                        fence_after();
                        issue_stage2(tmem, sE, sD + qh * 192 * 128, 0, 4);
                        mma_commit(barA);
                        ++nA;
                    }
                }
            }
            // the last of each, before shared memory and TMEM are given up (after
            // an expired wait, the drainers' too: they see MMAs come in late)
            mbar_wait(barD, (nD - 1u) & 1u);
            mbar_wait(barY, (nY - 1u) & 1u);
            if (nP) mbar_wait(barP, (nP - 1u) & 1u);
            if (nA) mbar_wait(barA, (nA - 1u) & 1u);
        }
    } else {
        const int quarter = warp & 3, cg = warp >> 2;
        const int row = quarter * 32 + lane;
        const uint32_t lane_base = tmem + ((uint32_t)(quarter * 32) << 16);
        const int k = row & 63;                                   // stage 1: row of a class
        const int p = 2 * (8 * (row >> 4) + (row & 7)) + ((row >> 3) & 1);     // stage 2: M index -> p
        uint32_t phA = 0, phY = 0;
        uint32_t T[8][4];
        auto wait = [&](uint32_t bar, uint32_t &phase) {
            ok = __all_sync(0xffffffffu, mbar_wait(bar, phase)) && ok;
            phase ^= 1u;
            fence_after();
            return ok;
        };
        // this warp's reads of tensor memory and writes of shared memory are done
        auto done = [&]() {
            fence_before();
            fence_async();
            __syncwarp();
            if (lane == 0)
                asm volatile("mbarrier.arrive.release.cta.shared::cta.b64 _, [%0];" ::"r"(barC) : "memory");
        };
        auto finish = [&](long long leaf, int cls, int qh) {
            float2 *out = c0 + leaf * M + (2 * (32 * qh + 8 * cg) + cls) * b + p;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const df v = biased_to_df(T[j][0], T[j][1], T[j][2], T[j][3]);
                out[2 * j * b] = make_float2(v.hi, v.lo);
            }
        };
        long long pending = -1;
        for (long long leaf = blockIdx.x; ok && leaf < count; leaf += gridDim.x) {
            if (!wait(barY, phY)) break;
            // rows m and 127 - m, two 16-byte chunks a thread
            for (int o = tid; o < 1024; o += 512) {
                const int kh = o >> 9, m = (o >> 3) & 63, j = o & 7;
                unsigned char *t = gbase + kOffY128 + kh * 128 * 128;
                fold_chunks(reinterpret_cast<uint4 *>(t + m * 128 + ((j ^ (m & 7)) << 4)),
                            reinterpret_cast<uint4 *>(t + (127 - m) * 128 + ((j ^ (7 - (m & 7))) << 4)));
            }
            done();
            if (pending >= 0) finish(pending, 1, 1);
            for (int cls = 0; cls < 2 && ok; ++cls) {
                // ---- stage 1 and the digits, the p of parity 1 - cls, then of cls
                for (int turn = 0; turn < 2; ++turn) {
                    const int a = turn ? cls : 1 - cls;
                    if (!wait(barA, phA)) break;
                    if ((quarter >> 1) == cls) {
#pragma unroll 1
                        for (int h = 0; h < 2; ++h) {
                            // p' = 16 cg + 8 h + (0 .. 7)
                            uint32_t z[2][4][2];
#pragma unroll
                            for (int g = 0; g < 2; ++g) {
                                uint32_t v[6][4];
#pragma unroll
                                for (int sd = 0; sd < 6; ++sd)
                                    tmem_ld4(lane_base + 192 * (cg >> 1) + 32 * sd + 16 * (cg & 1) + 8 * h + 4 * g, v[sd]);
                                wait_ld();
#pragma unroll
                                for (int i = 0; i < 4; ++i) {
                                    const unsigned long long x =
                                        join_digits(v[0][i], v[1][i], v[2][i], v[3][i], v[4][i], v[5][i],
                                                    cls ? 0ull : cen[2 * (16 * cg + 8 * h + 4 * g + i) + a]);
                                    z[g][i][0] = (uint32_t)x;
                                    z[g][i][1] = (uint32_t)(x >> 32);
                                }
                            }
                            const int chunk = 2 * (2 * cg + h) + a;
                            unsigned char *dst = gbase + kOffE128 + (chunk >> 3) * kTileE + k * 128 +
                                                 (((chunk & 7) ^ (k & 7)) << 4);
#pragma unroll
                            for (int t = 0; t < 8; ++t) {
                                const int w = t >> 2, y = t & 3;
                                *reinterpret_cast<uint4 *>(dst + t * 2 * kTileE) =
                                    make_uint4(bytes_less_128(z[0][0][w], z[0][1][w], y),
                                               bytes_less_128(z[0][2][w], z[0][3][w], y),
                                               bytes_less_128(z[1][0][w], z[1][1][w], y),
                                               bytes_less_128(z[1][2][w], z[1][3][w], y));
                            }
                        }
                    }
                    done();
                }
                // ---- stage 2
                for (int qh = 0; qh < 2 && ok; ++qh) {
                    if (!wait(barA, phA)) break;
                    drain_diagonals(lane_base, 8 * cg, T);
                    if (qh == 0 || cls == 0) {
                        done();
                        finish(leaf, cls, qh);
                    }
                }
            }
            pending = leaf;
        }
        if (ok && pending >= 0) finish(pending, 1, 1);
    }
    fence_before();
    const bool all_ok = __syncthreads_and(ok) != 0;
    if (tid == 0 && !all_ok && ctr) raise_error(ctr, kDevErrTimeout, 13u);
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
}

bool corr_sep_tc_available(int b, int) { return b == septc::kB || b == 128; }

cudaError_t launch_corr_sep_tc(const CorrArgs &a, cudaStream_t st) {
    const DictDev &d = *a.d;
    if (!corr_sep_tc_available(d.b, d.nf) || !d.tmap_sepd || !a.tmap_Ysep) return cudaErrorInvalidValue;
    const long long rows = a.count ? (long long)a.capacity : a.fixed_count;
    if (rows <= 0) return cudaSuccess;
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    if (d.b == 128) {
        if (d.fam0 != 0 || a.fmask != 1) return cudaErrorInvalidValue;            // the DCT-II family alone
        e = cudaFuncSetAttribute(corr_sep_tc128_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 septc::kSmemBytes128);
        if (e != cudaSuccess) return e;
        corr_sep_tc128_kernel<<<(unsigned)(rows < sms ? rows : sms), septc::kThreads128, septc::kSmemBytes128, st>>>(
            *reinterpret_cast<const CUtensorMap *>(a.tmap_Ysep), *reinterpret_cast<const CUtensorMap *>(d.tmap_sepd),
            d.nf * 128 * 128, d.Rs, a.count, a.fixed_count, a.c0, a.ctr);
        return cudaGetLastError();
    }
    const long long pairs = (rows + 1) / 2;
    const unsigned grid = (unsigned)(pairs < sms ? pairs : sms);
    e = cudaFuncSetAttribute(corr_sep_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, septc::kSmemBytes);
    if (e != cudaSuccess) return e;
    const int n = septc::kB * septc::kB, fmask = a.fmask ? a.fmask : 3;
    for (int f = 0; f < d.nf && e == cudaSuccess; ++f) {
        const int F = d.nf == 2 ? f : d.fam0;
        if (!((fmask >> F) & 1)) continue;
        corr_sep_tc_kernel<<<grid, septc::kThreads, septc::kSmemBytes, st>>>(
            *reinterpret_cast<const CUtensorMap *>(a.tmap_Ysep), *reinterpret_cast<const CUtensorMap *>(d.tmap_sepd), F,
            d.nf * n, f * n, d.Rs, a.count, a.fixed_count, a.c0, a.ctr);
        e = cudaGetLastError();
    }
    return e;
}

}  // namespace aqmp
