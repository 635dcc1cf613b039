// corr_sep.cu -- (a2) initial correlation with the separable fixed-point
// dictionary (sep.cuh) on the integer SIMT pipes: exact, and the reference
// twin of the tensor-core kernel of corr_sep_tc.cu (same bits).
//
// Section 2.2 step (b) needs <r0, phi_j> for every atom j.  The DCT-II and
// Haar atoms are outer products of 1-D rows (Section 2.1), so the M = 2 b^2
// correlations of a block are B Y B^T for each family: two b x b x b products
// instead of the b^4 per family of a dense D^T y, and the rows' structure
// (the DCT-II rows' mirror symmetry, the Haar rows' two constant halves)
// cuts that further, as the kernel below describes.  In integers:
//   stage 1  Z~[p][m] = sum_i Bf[p][i] y~[i][m]   (48-bit x 8-bit -> int64)
//   stage 2  T~[p][q] = sum_m Bf[q][m] Z~[p][m]   (48-bit x 59-bit -> int128)
// Bf is held as 24-bit limbs (lo in [-2^23, 2^23), hi = (Bf - lo) / 2^24,
// |hi| < 2^23.5), and the stage-1 results (Z~+-, below, |Z~+-| < 2^60) as
// two 32-bit ones (zl in [-2^31, 2^31), zh = (z - zl) / 2^32, |zh| < 2^28),
// so every partial product is one 32 x 32 -> 64-bit multiply-add, at most
// 2^54.5 in magnitude, and each of the four limb sums over at most b/2 = 64
// terms stays below 2^61.
#include <cuda_runtime.h>
#include <cuda_bf16.h>

#include "common.cuh"
#include "kernels.h"
#include "sep.cuh"

namespace aqmp {

namespace {

constexpr int ilog2(int x) { return x <= 1 ? 0 : 1 + ilog2(x / 2); }

// Leaves per CTA: enough for 4096 outputs per family and stage.
template <int B>
constexpr int sep_group() { return B >= 64 ? 1 : 4096 / (B * B); }

// Z~ split into balanced limbs: z = zl + zh 2^32.
struct Limbs2 {
    int32_t zl, zh;
};

__device__ __forceinline__ Limbs2 split2(long long z) {
    const int32_t zl = (int32_t)(uint32_t)(unsigned long long)z;    // z mod 2^32, in [-2^31, 2^31)
    return Limbs2{zl, (int32_t)((z - (long long)zl) >> 32)};
}

__device__ __forceinline__ long long mul_wide(int32_t a, int32_t b) { return (long long)a * (long long)b; }

}  // namespace

// Threads per CTA: at side 128 the leaf's shared memory (181 KB, most of it
// Z~+-) leaves room for one CTA per SM, so that CTA takes 768 threads to hide
// the latency of its loads; 256 elsewhere.
template <int B>
constexpr int sep_threads() { return B >= 128 ? 768 : 256; }

// Shared-memory layout of one CTA (G leaves): the centred pixels, their
// even and odd column halves, and the Z~ region, which the Haar pass reuses.
// A Haar-only launch (HO) keeps that pass's arrays alone.
template <int B, bool HO = false>
struct SepSmem {
    static constexpr int n = B * B, H = B / 2, G = sep_group<B>();
    static constexpr int RS = B + 1;                           // row stride of Z~+- and of the table
    static constexpr int YS = B + 4;                           // row stride of the pixels (bytes): the
                                                               // transposing stores hit distinct banks
    static constexpr size_t yt = 0;                            // int8  [G][i][YS]
    static constexpr size_t ys = HO ? 0 : (G * B * YS + 15) & ~15;      // int16 [G][parity][i < H][m]
    static constexpr size_t z = ys + (HO ? 0 : ((2 * G * n + 15) & ~15));   // Limbs2 [G][p][RS] / int [G][RS][RS]
    // the Haar pass: K [G][p][RS] (int), the first transform [G][p][DS] (int16), sums of 16 values [c][G * B] (int)
    static constexpr int CH = B < 16 ? B : 16, C = B / CH, DS = B + 2;
    static constexpr size_t d1 = sizeof(int) * G * B * RS, part = d1 + ((sizeof(int16_t) * G * B * DS + 15) & ~15),
                            hbytes = part + (C > 1 ? sizeof(int) * C * G * B : 0);
    static constexpr size_t zbytes = HO ? ((hbytes + 15) & ~15) : sizeof(Limbs2) * G * B * RS;
    static constexpr int E = 1 + ilog2(B);                     // Haar scale classes: row 0, scales 1 .. b/2
    static constexpr size_t ptab = z + zbytes;                 // int4 [E][E]: the limbs of -fL(c1) fL(c2)
    static constexpr size_t bytes = ptab + sizeof(int4) * E * E;
    static_assert(hbytes <= sizeof(Limbs2) * G * B * RS, "the Haar pass fits the Z~ region");
};

__device__ __forceinline__ long long bf_value(int2 w) { return (long long)w.y * (1ll << 24) + w.x; }

// The Haar class of a row: 0 for row 0, 1 + log2 of the scale's first row.
__device__ __forceinline__ int haar_class(int r) { return 32 - __clz(r); }

// Unnormalised Haar transform (row 0 the sum, row r >= 1 the sum over its
// first half minus that over its second) of CH values in v, in place of a
// part of a longer row: put(level row offset, value) for all but the sum,
// which is returned.  c is the part's number of C: the rows of scale s that
// lie in the part are B / s + c CH / s + t.
template <int B, int CH, typename V, typename Put>
__device__ __forceinline__ V haar_part(V (&v)[CH], int c, Put put) {
#pragma unroll
    for (int s = 2; s <= CH; s *= 2) {
#pragma unroll
        for (int t = 0; t < CH / s; ++t) {
            const V x = v[2 * t], y = v[2 * t + 1];
            put(B / s + c * (CH / s) + t, x - y);
            v[t] = x + y;
        }
    }
    return v[0];
}

// Row r < C of the transform from the C parts' sums at s[0], s[stride], ...
template <int C>
__device__ __forceinline__ int haar_join(const int *s, int stride, int r) {
    const int len = r == 0 ? C : C >> (31 - __clz(r));           // parts under the row
    const int at = r == 0 ? 0 : (r - (1 << (31 - __clz(r)))) * len;
    int sum = 0;
    for (int i = 0; i < len; ++i) {
        const int x = s[(at + i) * stride];
        sum += r != 0 && 2 * i >= len ? -x : x;
    }
    return sum;
}

// One CTA handles G leaves at a time (grid-stride over the leaves).
//
// DCT-II family: row p of Bf equals (-1)^p times its mirror image, so with
// the column halves y+-[i][m] = y~[i][m] +- y~[b-1-i][m] (i < b/2) stage 1
// needs b/2 terms, and stage 1 stores Z~+-[p][m] = Z~[p][m] +- Z~[p][b-1-m]
// (m < b/2), of which stage 2 takes Z~+ for even q and Z~- for odd q, again
// over b/2 terms: half the multiply-adds of the plain products, the same
// exact integers.  |Z~+-| < 2^60, so zh < 2^28 and every limb sum over
// b/2 <= 64 terms stays below 2^61.
//
// Haar family: row p of Bf is +fL on its first half and -fL on its second
// (row 0: fL throughout), and fL depends only on the row's scale.  So
// T~[p][q] = fL(p) fL(q) K[p][q] with K the integer 2-D Haar transform of y~
// (|K| <= 2^21): one pass of sums and differences along i, one along m, two
// additions per value each, in parts of 16 per thread.  The products
// fL(c1) fL(c2) of the 1 + log2 b scale classes are formed once per CTA and
// kept negated in three signed 32-bit limbs (2^95 fits with that sign), so
// T + the rounding's bias is a chain of three 32-bit multiply-adds.  The
// integer work of an output is now the smaller part of it beside the rounding.
// Side 64, 50 910 leaves, this family alone: 1.88 -> 0.85 ms (a summed-area
// table, nine reads and an int128 product per output, before).
template <int B, bool HO>
__global__ void __launch_bounds__(sep_threads<B>())
corr_sep_simt_kernel(int nf, int fam0, int fmask, int Kpad, const int2 *__restrict__ Bs, const int2 *__restrict__ BsT,
                     const long long *__restrict__ Rs, const __nv_bfloat16 *__restrict__ Y,
                     const unsigned *count_dev, long long fixed_count, float2 *__restrict__ c0) {
    using L = SepSmem<B, HO>;
    constexpr int n = L::n, H = L::H, G = L::G, RS = L::RS, YS = L::YS;
    if (HO) fmask &= 2;                                       // the Haar family alone
    constexpr int PT = 4;                                     // p values per thread in DCT stage 2
    static_assert(B >= PT && B % PT == 0, "side");
    extern __shared__ __align__(16) unsigned char smem[];
    int8_t *yt = reinterpret_cast<int8_t *>(smem + L::yt);
    int16_t *ys = reinterpret_cast<int16_t *>(smem + L::ys);
    Limbs2 *Z = reinterpret_cast<Limbs2 *>(smem + L::z);

    constexpr int nt = sep_threads<B>(), E = L::E;
    int4 *ptab = reinterpret_cast<int4 *>(smem + L::ptab);

    const long long count = count_dev ? (long long)*count_dev : fixed_count;
    const int M = nf * n;
    const int tid = threadIdx.x;
    if ((nf == 2 || fam0 == 1) && ((fmask >> 1) & 1)) {
        // the class products
        const int2 *Bh = Bs + (size_t)n;
        for (int e = tid; e < E * E; e += nt) {
            const int c1 = e / E, c2 = e - c1 * E;
            const int r1 = c1 == 0 ? 0 : 1 << (c1 - 1), r2 = c2 == 0 ? 0 : 1 << (c2 - 1);   // first row of the class
            const __int128 P = -(__int128)bf_value(Bh[r1 * B]) * bf_value(Bh[r2 * B]);
            const int32_t l0 = (int32_t)(uint32_t)(unsigned __int128)P;
            const long long P1 = (long long)((P - l0) >> 32);
            const int32_t l1 = (int32_t)(uint32_t)(unsigned long long)P1;
            ptab[e] = make_int4(l0, l1, (int32_t)((P1 - l1) >> 32), 0);
        }
        __syncthreads();
    }
    for (long long base = (long long)blockIdx.x * G; base < count; base += (long long)gridDim.x * G) {
        const int live = (int)min((long long)G, count - base);
        if constexpr (!HO) {
            // centred pixels, transposed so that the contractions read consecutive m
            for (int o = tid; o < G * n; o += nt) {
                const int g = o / n, v = o - g * n;
                const int m = v / B, i = v - m * B;
                int8_t y = 0;
                if (g < live) y = (int8_t)__bfloat162float(Y[(base + g) * Kpad + v]);
                yt[(g * B + i) * YS + m] = y;
            }
            __syncthreads();
        }
        for (int f = 0; f < nf; ++f) {
            const int F = nf == 2 ? f : fam0;
            if (!((fmask >> F) & 1)) continue;                   // uniform
            const int2 *Bf = Bs + (size_t)F * n;
            const long long *R = Rs + F * B;
            float2 *out = c0 + (nf == 2 ? f * n : 0);
            if (F == 0) {
                if constexpr (!HO) {
                const int2 *BfT = BsT + (size_t)F * n;
                for (int o = tid; o < G * H * B; o += nt) {
                    const int g = o / (H * B), r = o - g * (H * B);
                    const int i = r / B, m = r - i * B;
                    const int a = yt[(g * B + i) * YS + m], c = yt[(g * B + B - 1 - i) * YS + m];
                    ys[(2 * g) * H * B + r] = (int16_t)(a + c);
                    ys[(2 * g + 1) * H * B + r] = (int16_t)(a - c);
                }
                __syncthreads();
                // stage 1: Z~[p][m] and Z~[p][b-1-m] together, m < b/2 across threads
                for (int o = tid; o < G * B * H; o += nt) {
                    const int g = o / (B * H), r = o - g * (B * H);
                    const int p = r / H, m = r - p * H;
                    const int16_t *yp = ys + (2 * g + (p & 1)) * H * B;
                    long long lo1 = 0, hi1 = 0, lo2 = 0, hi2 = 0;
#pragma unroll 8
                    for (int i = 0; i < H; ++i) {
                        const int2 w = Bf[p * B + i];
                        const int32_t a = yp[i * B + m], c = yp[i * B + B - 1 - m];
                        lo1 += mul_wide(w.x, a);
                        hi1 += mul_wide(w.y, a);
                        lo2 += mul_wide(w.x, c);
                        hi2 += mul_wide(w.y, c);
                    }
                    const long long z1 = hi1 * (1ll << 24) + lo1, z2 = hi2 * (1ll << 24) + lo2;
                    Limbs2 *zr = Z + (g * B + p) * RS;
                    zr[m] = split2(z1 + z2);
                    zr[H + 1 + m] = split2(z1 - z2);
                }
                __syncthreads();
                // stage 2: T~[g][p][q], q lane-fastest, PT consecutive p per thread
                for (int o = tid; o < G * n / PT; o += nt) {
                    const int g = o / (n / PT), r = o - g * (n / PT);
                    const int q = r % B, p0 = (r / B) * PT;
                    const Limbs2 *zr = Z + (g * B + p0) * RS + ((q & 1) ? H + 1 : 0);
                    long long a0[PT], a1[PT], a2[PT], a3[PT];
#pragma unroll
                    for (int k = 0; k < PT; ++k) a0[k] = a1[k] = a2[k] = a3[k] = 0;
#pragma unroll 4
                    for (int m = 0; m < H; ++m) {
                        const int2 w = BfT[m * B + q];                 // Bf[q][m]: (lo, hi)
#pragma unroll
                        for (int k = 0; k < PT; ++k) {
                            const Limbs2 z = zr[k * RS + m];
                            a0[k] += mul_wide(w.x, z.zl);              // weight 1
                            a1[k] += mul_wide(w.y, z.zl);              // 2^24
                            a2[k] += mul_wide(w.x, z.zh);              // 2^32
                            a3[k] += mul_wide(w.y, z.zh);              // 2^56
                        }
                    }
                    if (g < live) {
                        float v[2 * PT];
#pragma unroll
                        for (int k = 0; k < PT; ++k) {
                            __int128 T = (__int128)a3[k] * ((__int128)1 << 56) + (__int128)a2[k] * ((__int128)1 << 32) +
                                         (__int128)a1[k] * ((__int128)1 << 24) + (__int128)a0[k];
                            T += (__int128)(128ll * R[p0 + k]) * R[q];
                            const df c = int128_to_df(T);
                            v[2 * k] = c.hi;
                            v[2 * k + 1] = c.lo;
                        }
                        float4 *dst = reinterpret_cast<float4 *>(out + (base + g) * M + q * B + p0);
#pragma unroll
                        for (int k = 0; k < PT / 2; ++k)
                            dst[k] = make_float4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
                    }
                }
                }
            } else {
                constexpr int CH = L::CH, C = L::C, DS = L::DS, rows = G * B;
                int *K = reinterpret_cast<int *>(smem + L::z);                       // [G][p][RS]
                int16_t *D1 = reinterpret_cast<int16_t *>(smem + L::z + L::d1);      // [G][p][DS]
                int *part = reinterpret_cast<int *>(smem + L::z + L::part);
                // along i, straight from the gathered pixels (y~ at m b + i), in
                // exact floats: lanes take consecutive m
                for (int o = tid; o < rows * C; o += nt) {
                    const int row = o % rows, c = o / rows, g = row / B, m = row % B;
                    uint32_t x[CH / 2] = {};
                    if (g < live) {
                        const __nv_bfloat16 *src = Y + (base + g) * Kpad + m * B + c * CH;
                        if constexpr (CH == 4) {
                            const uint2 u = *reinterpret_cast<const uint2 *>(src);
                            x[0] = u.x, x[1] = u.y;
                        } else {
#pragma unroll
                            for (int w = 0; w < CH / 8; ++w) {
                                const uint4 u = reinterpret_cast<const uint4 *>(src)[w];
                                x[4 * w] = u.x, x[4 * w + 1] = u.y, x[4 * w + 2] = u.z, x[4 * w + 3] = u.w;
                            }
                        }
                    }
                    float v[CH];
#pragma unroll
                    for (int w = 0; w < CH / 2; ++w) {
                        v[2 * w] = __uint_as_float(x[w] << 16);
                        v[2 * w + 1] = __uint_as_float(x[w] & 0xffff0000u);
                    }
                    int16_t *dst = D1 + g * B * DS + m;
                    auto as_int = [](float f) { return __float_as_int(__fadd_rn(f, 12582912.0f)); };   // + 0x4B400000
                    const float sum = haar_part<B, CH>(v, c, [&](int p, float f) { dst[p * DS] = (int16_t)as_int(f); });
                    if (C > 1) part[c * rows + row] = as_int(sum) - 0x4B400000;
                    else dst[0] = (int16_t)as_int(sum);
                }
                if (C > 1) {
                    __syncthreads();
                    for (int o = tid; o < rows * C; o += nt) {
                        const int row = o % rows, r = o / rows;
                        D1[((row / B) * B + r) * DS + row % B] = (int16_t)haar_join<C>(part + row, rows, r);
                    }
                }
                __syncthreads();
                // along m: lanes take consecutive p
                for (int o = tid; o < rows * C; o += nt) {
                    const int row = o % rows, c = o / rows;
                    const int32_t *src = reinterpret_cast<const int32_t *>(D1 + row * DS + c * CH);
                    int *dst = K + row * RS;
                    int v[CH];
#pragma unroll
                    for (int w = 0; w < CH / 2; ++w) {
                        const int x = src[w];
                        v[2 * w] = (int)(int16_t)x;
                        v[2 * w + 1] = x >> 16;
                    }
                    const int sum = haar_part<B, CH>(v, c, [&](int q, int x) { dst[q] = x; });
                    if (C > 1) part[c * rows + row] = sum;
                    else dst[0] = sum;
                }
                __syncthreads();
                if (C > 1) {
                    for (int o = tid; o < rows * C; o += nt)
                        K[(o % rows) * RS + o / rows] = haar_join<C>(part + o % rows, rows, o / rows);
                    __syncthreads();
                }
                // T[g][p][q], p lane-fastest and the same in every turn of a thread
                const int p = tid % B, cp = haar_class(p) * E;
                for (int o = tid; o < G * n; o += nt) {
                    const int q = o / B % B, g = o / n;
                    int k = -K[(g * B + p) * RS + q];
                    if ((p | q) == 0) k -= 128 * n;             // centring: rows r >= 1 sum to zero, R[0] = b fL(0)
                    const int4 l = ptab[cp + haar_class(q)];
                    const long long x0 = mul_wide(l.x, k) + (long long)kDigitBiasLo;
                    const long long x1 = mul_wide(l.y, k) + (x0 >> 32);
                    const long long x2 = mul_wide(l.z, k) + (long long)kDigitBiasHi + (x1 >> 32);
                    if (g < live) {
                        const df c = biased_to_df((uint32_t)x0, (uint32_t)x1, (uint32_t)x2, (uint32_t)(x2 >> 32));
                        out[(base + g) * M + q * B + p] = make_float2(c.hi, c.lo);
                    }
                }
            }
            __syncthreads();
        }
    }
}

template <int B, bool HO>
static cudaError_t launch_sep_simt_t(const CorrArgs &a, cudaStream_t st) {
    constexpr int G = sep_group<B>();
    const size_t smem = SepSmem<B, HO>::bytes;
    auto kern = corr_sep_simt_kernel<B, HO>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, sep_threads<B>(), smem);
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    long long need = ((long long)a.capacity + G - 1) / G;
    long long grid = (long long)sms * (per_sm < 1 ? 1 : per_sm);
    if (need < grid) grid = need;
    if (grid < 1) grid = 1;
    const DictDev &d = *a.d;
    kern<<<(unsigned)grid, sep_threads<B>(), smem, st>>>(d.nf, d.fam0, a.fmask ? a.fmask : 3, d.Kpad, d.Bs, d.BsT,
                                                          d.Rs, a.Y, a.count,
                                                          a.fixed_count, a.c0);
    return cudaGetLastError();
}

cudaError_t launch_corr_sep_simt(const CorrArgs &a, cudaStream_t st) {
    // the Haar family alone gets its own instantiation: no DCT-II code or
    // shared memory, so more CTAs fit on an SM
    const DictDev &d = *a.d;
    const bool ho = a.fmask == 2 || (d.nf == 1 && d.fam0 == 1);
    switch (d.b) {
        case 4: return ho ? launch_sep_simt_t<4, true>(a, st) : launch_sep_simt_t<4, false>(a, st);
        case 8: return ho ? launch_sep_simt_t<8, true>(a, st) : launch_sep_simt_t<8, false>(a, st);
        case 16: return ho ? launch_sep_simt_t<16, true>(a, st) : launch_sep_simt_t<16, false>(a, st);
        case 32: return ho ? launch_sep_simt_t<32, true>(a, st) : launch_sep_simt_t<32, false>(a, st);
        case 64: return ho ? launch_sep_simt_t<64, true>(a, st) : launch_sep_simt_t<64, false>(a, st);
        case 128: return ho ? launch_sep_simt_t<128, true>(a, st) : launch_sep_simt_t<128, false>(a, st);
    }
    return cudaErrorInvalidValue;
}

}  // namespace aqmp
