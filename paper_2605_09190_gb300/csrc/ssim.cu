// ssim.cu -- the mean SSIM of Section 3 and its gradient with respect to the
// reconstruction, for up to kRefinePlanes images in one launch of each pass.
//
// SSIM over the valid region with an 11 x 11 Gaussian window w = g g^T
// (sigma 1.5), K1 = 0.01, K2 = 0.03, L = 255.  Per window, with the window
// means mx, my, Exy = E[x y] and Ed = E[(x - y)^2]:
//   A1 = 2 mx my + C1, B1 = A1 + (mx - my)^2 = mx^2 + my^2 + C1,
//   A2 = 2 (Exy - mx my) + C2,
//   B2 = A2 + (Ed - (mx - my)^2) = var x + var y + C2,
//   f = A1 A2 / (B1 B2).
// Ed in the place of E[x^2 + y^2]: an error of Exy, the larger one, then moves
// A2 and B2 together, and f by 1 - A2 / B2 of it alone.
// With S = mean f over the N windows, for a pixel k of y:
//   dS/dy[k] = (1/N) sum_win w(k - win) (f_my + 2 y[k] f_Eyy + x[k] f_Exy),
//   f_my = f (2 mx / A1 - 2 mx / A2 - 2 my / B1 + 2 my / B2),
//   f_Exy = 2 f / A2,   f_Eyy = -f / B2,
// i.e. the per-window partials filtered back with the (symmetric, separable)
// window.
//
// Everything is double-float (~2^-46 relative, so that E[s] - mu^2 keeps the
// variance; pixels beyond any image's take the window formula in FP64) on the packed FP32 pipes: GB300's FP64 rate is 1/64 of its FP32
// rate, and the window formula in FP64 alone took a third of the former
// window pass.  An 11-tap pass keeps each sum as (s, c): s the running FP32
// sum, c the sum of the exact errors of its products and additions and of the
// low words' terms, joined once at the end (Ogita, Rump and Oishi's Dot2
// scheme) -- 12 operations a tap, against 15 with a renormalised pair.  A
// product's small terms meet before they meet c, and taps come smallest weights
// first where the order is free, so that few roundings are of c's size.
// Error of a window's value against long double, root mean square, of
// renormalised pairs with E[x^2], E[y^2], E[x y] and the formula in FP64, and
// here: 3.1e-12 and 0.8e-12 for a piecewise scene with noise of 4 grey values,
// 3.0e-12 and 0.1e-12 with 1, 1.0e-12 and 0.6e-12 for a gradient one with 8,
// 1.6e-14 and 1.5e-14 for two independent images.
//
// Forward: a CTA loads the pixels of a tile of windows once, filters the four
// fields x, y, x y, (x - y)^2 along the rows into shared memory and down the
// columns into registers, and writes the three partials (24 bytes a window);
// backward: the same with the partials' tile, columns first.  Bound by the
// FP32 pipes (about 154 taps a pixel); the four passes over global memory
// with 40-byte intermediates that this replaces were bound by memory latency.
// 16 planes of 512x512, forward and gradient: 2.2 ms in 64 launches -> 225 us
// forward and 203 us backward.
#include <cuda_runtime.h>

#include "common.cuh"
#include "f32x2.cuh"
#include "kernels.h"

namespace aqmp {

namespace {

constexpr int kThreads = 256;
constexpr int kTW = 32;                       // windows / pixels across a tile
constexpr int kCols = kTW + 10;               // with the halo

struct Acc2 {
    f2 s, c;
};

struct Acc1 {
    float s, c;
};

// acc + g (v + vl) for two sums at once, g = gh - ngl, ngh = -gh.
template <bool LO>
__device__ __forceinline__ void tap(Acc2 &a, f2 gh, f2 ngh, f2 ngl, f2 v, f2 vl) {
    const f2 p = f2_mul(gh, v);
    f2 ne = f2_fma(ngh, v, p);                                  // gh v = p - ne exactly
    if (LO) ne = f2_fma(ngh, vl, ne);
    ne = f2_fma(ngl, v, ne);
    const f2 s = f2_add(a.s, p);
    const f2 bb = f2_sub(s, a.s);
    const f2 t = f2_add(f2_sub(a.s, f2_sub(s, bb)), f2_sub(p, bb));
    a.c = f2_add(a.c, f2_sub(t, ne));
    a.s = s;
}

__device__ __forceinline__ void tap(Acc1 &a, float gh, float ngh, float ngl, float v, float vl) {
    const float p = __fmul_rn(gh, v);
    const float ne = __fmaf_rn(ngl, v, __fmaf_rn(ngh, vl, __fmaf_rn(ngh, v, p)));
    const df s = df_two_sum(a.s, p);
    a.c = __fadd_rn(a.c, __fsub_rn(s.lo, ne));
    a.s = s.hi;
}

__device__ __forceinline__ df join(float s, float c) { return df_fast_two_sum(s, c); }

// 1 / d to ~2^-46 for a normal d.
__device__ __forceinline__ df df_recip(df d) {
    const float r = __frcp_rn(d.hi);
    const float e = __fmaf_rn(-d.lo, r, __fmaf_rn(-d.hi, r, 1.0f));       // 1 - d r
    return df_fast_two_sum(r, __fmul_rn(r, __fmaf_rn(e, e, e)));
}

__device__ __forceinline__ df twice(df a) { return df_scale(a, 2.0f); }

__host__ __device__ __forceinline__ df df_split(double v) {
    const float hi = (float)v;
    return df{hi, (float)(v - (double)hi)};
}

// A window's value and partials.
struct Window {
    df f, my, yy, xy;
};

// ... from its means in FP64, where 1 / (B1 B2) and its low word would leave
// the range of FP32: B1 or B2 above 2^48, pixels of 10^7 and more.  Out of
// line, since no image has such pixels (a refinement that diverges does).
__device__ __noinline__ void window_fp64(df mx_, df my_, df exy_, df ed_, Window *out) {
    const double mx = df_to_double(mx_), my = df_to_double(my_), exy = df_to_double(exy_), ed = df_to_double(ed_);
    const double C1 = (0.01 * 255.0) * (0.01 * 255.0), C2 = (0.03 * 255.0) * (0.03 * 255.0);
    const double mxy = mx * my, ee = (mx - my) * (mx - my);
    const double A1 = 2.0 * mxy + C1, A2 = 2.0 * (exy - mxy) + C2, iB1 = 1.0 / (A1 + ee), iB2 = 1.0 / (A2 + (ed - ee));
    const double t1 = A2 * iB1 * iB2, t2 = A1 * iB1 * iB2, f = A1 * t1;          // f / A1, f / A2
    out->f = df_split(f);
    out->my = df_split(2.0 * mx * (t1 - t2) - 2.0 * my * f * (iB1 - iB2));
    out->yy = df_split(-f * iB2);
    out->xy = df_split(2.0 * t2);
}

// The plane of this CTA's tile, and the tile's place in it.
__device__ __forceinline__ const SsimPlane &find_plane(const SsimArgs &a, int &ty, int &tx) {
    int i = 0;
    while (i + 1 < a.n && a.p[i + 1].tile0 <= blockIdx.x) ++i;
    const unsigned t = blockIdx.x - a.p[i].tile0;
    ty = (int)(t / a.p[i].tiles_x);
    tx = (int)(t - (unsigned)ty * a.p[i].tiles_x);
    return a.p[i];
}

// Tile heights: RV output rows per thread in the column pass, eight threads
// to a column.
template <int RV>
struct FwdTile {
    static constexpr int HR = RV == 7 ? 64 : 32;              // pixel rows of the tile
    static constexpr int TH = HR - 10;                        // window rows
    static constexpr int XW = 44;                             // pixel row stride
    static constexpr int PAD = 8 * RV + 10 - HR;              // rows past the tile that the column pass reads, unused
    static constexpr size_t bytes = sizeof(float2) * HR * XW + sizeof(float4) * (2 * HR + PAD) * kTW;
    static_assert(8 * RV >= TH && PAD >= 0 && PAD < HR, "rows");
};

template <int RV>
__global__ void __launch_bounds__(kThreads, 2) ssim_forward_kernel(const __grid_constant__ SsimArgs a) {
    using T = FwdTile<RV>;
    extern __shared__ __align__(16) unsigned char smem[];
    float2 *xy = reinterpret_cast<float2 *>(smem);                        // [HR][XW] (x, y)
    float4 *Hm = reinterpret_cast<float4 *>(xy + T::HR * T::XW);           // [HR][TW] x, y: high words, low words
    float4 *Hp = Hm + T::HR * kTW;                                         // [HR][TW] x y, (x - y)^2
    int ty, tx;
    const SsimPlane &P = find_plane(a, ty, tx);
    const int r0 = ty * T::TH, c0 = tx * kTW, wo = P.w - 10, ho = P.h - 10;

    for (int i = threadIdx.x; i < T::HR * kCols; i += kThreads) {
        const int r = i / kCols, c = i - r * kCols;
        float2 v = make_float2(0.0f, 0.0f);
        if (r0 + r < P.h && c0 + c < P.w)
            v = make_float2(P.x[(long long)(r0 + r) * P.x_pitch + c0 + c], P.y[(long long)(r0 + r) * P.y_pitch + c0 + c]);
        xy[r * T::XW + c] = v;
    }
    __syncthreads();

    // rows: four neighbouring outputs a thread, each pixel's products once
    for (int i = threadIdx.x; i < T::HR * (kTW / 4); i += kThreads) {
        const int r = i / (kTW / 4), c = i % (kTW / 4) * 4;
        Acc2 m[4], p[4];
#pragma unroll
        for (int o = 0; o < 4; ++o) m[o] = p[o] = Acc2{0ull, 0ull};
        const ulonglong2 *row = reinterpret_cast<const ulonglong2 *>(xy + r * T::XW + c);
#pragma unroll
        for (int i = 0; i < 14; ++i) {
            // pairs of pixels from both ends, the middle last
            const int two_at = i & 2 ? 6 - (i >> 2) : i >> 2, k = 2 * two_at + (i & 1);
            const ulonglong2 two = row[two_at];
            const f2 v = k & 1 ? two.y : two.x;
            const float x = f2_x(v), y = f2_y(v);
            const df c2 = df_two_prod(x, y), d = df_two_sum(x, -y), dd = df_two_prod(d.hi, d.hi);
            const f2 ph = f2_make(c2.hi, dd.hi);
            const f2 pl = f2_make(c2.lo, __fmaf_rn(2.0f * d.hi, d.lo, dd.lo));
#pragma unroll
            for (int o = 0; o < 4; ++o) {
                const int j = k - o;
                if (j < 0 || j > 10) continue;
                tap<false>(m[o], a.gh[j], a.ngh[j], a.ngl[j], v, 0ull);
                tap<true>(p[o], a.gh[j], a.ngh[j], a.ngl[j], ph, pl);
            }
        }
#pragma unroll
        for (int o = 0; o < 4; ++o) {
            const df x = join(f2_x(m[o].s), f2_x(m[o].c)), y = join(f2_y(m[o].s), f2_y(m[o].c));
            const df s = join(f2_x(p[o].s), f2_x(p[o].c)), q = join(f2_y(p[o].s), f2_y(p[o].c));
            Hm[r * kTW + c + o] = make_float4(x.hi, y.hi, x.lo, y.lo);
            Hp[r * kTW + c + o] = make_float4(s.hi, q.hi, s.lo, q.lo);
        }
    }
    __syncthreads();

    // columns: RV consecutive outputs a thread
    const int col = threadIdx.x % kTW, row = threadIdx.x / kTW * RV;
    Acc2 m[RV], p[RV];
#pragma unroll
    for (int o = 0; o < RV; ++o) m[o] = p[o] = Acc2{0ull, 0ull};
#pragma unroll 1
    for (int i = 0; i < 11; ++i) {
        const int j = i & 1 ? 10 - (i >> 1) : i >> 1;                 // smallest weights first: 0, 10, 1, 9, ..., 5
        const f2 gh = a.gh[j], ngh = a.ngh[j], ngl = a.ngl[j];
        const int at = (row + j) * kTW + col;
#pragma unroll
        for (int o = 0; o < RV; ++o) {
            const ulonglong2 u = *reinterpret_cast<const ulonglong2 *>(Hm + at + o * kTW);
            const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(Hp + at + o * kTW);
            tap<true>(m[o], gh, ngh, ngl, u.x, u.y);
            tap<true>(p[o], gh, ngh, ngl, v.x, v.y);
        }
    }

    df sum{0.0f, 0.0f};
#pragma unroll
    for (int o = 0; o < RV; ++o) {
        const int r = r0 + row + o, c = c0 + col;
        if (row + o >= T::TH || r >= ho || c >= wo) continue;
        const df mx = join(f2_x(m[o].s), f2_x(m[o].c)), my = join(f2_y(m[o].s), f2_y(m[o].c));
        const df exy = join(f2_x(p[o].s), f2_x(p[o].c)), ed = join(f2_y(p[o].s), f2_y(p[o].c));
        const df mxy = df_mul(mx, my), e = df_sub(mx, my), ee = df_mul(e, e);
        const df A1 = df_add(twice(mxy), a.c1), B1 = df_add(A1, ee);
        const df A2 = df_add(twice(df_sub(exy, mxy)), a.c2), B2 = df_add(A2, df_sub(ed, ee));
        Window v;
        if (__builtin_expect(!(fmaxf(B1.hi, B2.hi) <= 0x1p48f), 0)) {
            Window big;
            window_fp64(mx, my, exy, ed, &big);
            v = big;
        } else {
            const df q = df_recip(df_mul(B1, B2));
            const df t1 = df_mul(A2, q), t2 = df_mul(A1, q);           // f / A1, f / A2
            v.f = df_mul(A1, t1);
            if (P.P4) {
                const df iB1 = df_mul(B2, q), iB2 = df_mul(B1, q);
                v.my = df_sub(df_mul(twice(mx), df_sub(t1, t2)), df_mul(df_mul(twice(my), v.f), df_sub(iB1, iB2)));
                v.yy = df_neg(df_mul(v.f, iB2));
                v.xy = twice(t2);
            }
        }
        sum = df_add(sum, v.f);
        if (P.P4) {
            const long long at = (long long)r * wo + c;
            P.P4[at] = make_float4(v.my.hi, v.yy.hi, v.my.lo, v.yy.lo);
            P.P2[at] = make_float2(v.xy.hi, v.xy.lo);
        }
    }
    // block sum, one atomic per block
    __shared__ double red[kThreads / 32];
    double local = df_to_double(sum);
    for (int off = 16; off > 0; off >>= 1) local += __shfl_xor_sync(0xffffffffu, local, off);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = local;
    __syncthreads();
    if (threadIdx.x == 0) {
        double v = 0.0;
        for (int i = 0; i < kThreads / 32; ++i) v += red[i];
        atomicAdd(P.sum, v / ((double)ho * (double)wo));
    }
}

// Rows per thread in the backward column pass, six threads to a column.
template <int RC>
struct BwdTile {
    static constexpr int HR = RC == 9 ? 64 : 32;              // window rows of the tile
    static constexpr int TH = HR - 10;                        // pixel rows
    static constexpr int RH = (TH + 7) / 8;                   // rows per thread in the row pass
    static constexpr size_t bytes = (sizeof(float4) + sizeof(float2)) * HR * kCols;
    static_assert(6 * RC >= TH && 6 * kCols <= kThreads, "rows");
};

template <int RC>
__global__ void __launch_bounds__(kThreads, 2) ssim_backward_kernel(const __grid_constant__ SsimArgs a) {
    using T = BwdTile<RC>;
    extern __shared__ __align__(16) unsigned char smem[];
    float4 *S4 = reinterpret_cast<float4 *>(smem);                        // [HR][kCols] f_my, f_Eyy
    float2 *S2 = reinterpret_cast<float2 *>(S4 + T::HR * kCols);           // [HR][kCols] f_Exy
    int ty, tx;
    const SsimPlane &P = find_plane(a, ty, tx);
    const int r0 = ty * T::TH, c0 = tx * kTW, wo = P.w - 10, ho = P.h - 10;

    // windows (r0 - 10 + r, c0 - 10 + c); none outside the valid region
    for (int i = threadIdx.x; i < T::HR * kCols; i += kThreads) {
        const int r = r0 - 10 + i / kCols, c = c0 - 10 + i % kCols;
        float4 u = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        float2 v = make_float2(0.0f, 0.0f);
        if (r >= 0 && r < ho && c >= 0 && c < wo) {
            u = P.P4[(long long)r * wo + c];
            v = P.P2[(long long)r * wo + c];
        }
        S4[i] = u;
        S2[i] = v;
    }
    __syncthreads();

    // columns: V[r][a] = sum_i g[i] P[r - i][a], kept in registers until the
    // tile has been read
    {
        const int col = threadIdx.x % kCols, row = threadIdx.x / kCols * RC;
        const bool on = threadIdx.x < 6 * kCols;
        Acc2 m[RC];
        Acc1 q[RC];
#pragma unroll
        for (int o = 0; o < RC; ++o) {
            m[o] = Acc2{0ull, 0ull};
            q[o] = Acc1{0.0f, 0.0f};
        }
        if (on) {
#pragma unroll 1
            for (int j = 0; j < 11; ++j) {
                const f2 gh = a.gh[j], ngh = a.ngh[j], ngl = a.ngl[j];
#pragma unroll
                for (int o = 0; o < RC; ++o) {
                    const int at = min(row + o + 10 - j, T::HR - 1) * kCols + col;
                    const ulonglong2 u = *reinterpret_cast<const ulonglong2 *>(S4 + at);
                    const float2 v = S2[at];
                    tap<true>(m[o], gh, ngh, ngl, u.x, u.y);
                    tap(q[o], f2_x(gh), f2_x(ngh), f2_x(ngl), v.x, v.y);
                }
            }
        }
        __syncthreads();
        if (on) {
#pragma unroll
            for (int o = 0; o < RC; ++o) {
                if (row + o >= T::TH) continue;
                const df y = join(f2_x(m[o].s), f2_x(m[o].c)), z = join(f2_y(m[o].s), f2_y(m[o].c));
                const df w = join(q[o].s, q[o].c);
                S4[(row + o) * kCols + col] = make_float4(y.hi, z.hi, y.lo, z.lo);
                S2[(row + o) * kCols + col] = make_float2(w.hi, w.lo);
            }
        }
        __syncthreads();
    }

    // rows, and the products: grad_y[r][c] = G1 + 2 y G2 + x G3 with
    // G[r][c] = sum_j g[j] V[r][c - j]
    const int col = threadIdx.x & 31, warp = threadIdx.x >> 5;
    Acc2 m[T::RH];
    Acc1 q[T::RH];
#pragma unroll
    for (int o = 0; o < T::RH; ++o) {
        m[o] = Acc2{0ull, 0ull};
        q[o] = Acc1{0.0f, 0.0f};
    }
#pragma unroll 1
    for (int j = 0; j < 11; ++j) {
        const f2 gh = a.gh[j], ngh = a.ngh[j], ngl = a.ngl[j];
#pragma unroll
        for (int o = 0; o < T::RH; ++o) {
            const int at = min(warp + 8 * o, T::HR - 1) * kCols + col + 10 - j;
            const ulonglong2 u = *reinterpret_cast<const ulonglong2 *>(S4 + at);
            const float2 v = S2[at];
            tap<true>(m[o], gh, ngh, ngl, u.x, u.y);
            tap(q[o], f2_x(gh), f2_x(ngh), f2_x(ngl), v.x, v.y);
        }
    }
#pragma unroll
    for (int o = 0; o < T::RH; ++o) {
        const int r = r0 + warp + 8 * o, c = c0 + col;
        if (warp + 8 * o >= T::TH || r >= P.h || c >= P.w) continue;
        const float xv = P.x[(long long)r * P.x_pitch + c], yv = P.y[(long long)r * P.y_pitch + c];
        df t = join(f2_x(m[o].s), f2_x(m[o].c));
        t = df_sub_mul(t, df{-2.0f * yv, 0.0f}, join(f2_y(m[o].s), f2_y(m[o].c)));
        t = df_sub_mul(t, df{-xv, 0.0f}, join(q[o].s, q[o].c));
        t = df_mul(t, P.scale);
        P.grad[(long long)r * P.grad_pitch + c] = ldexpf(__fadd_rn(t.hi, t.lo), P.scale_exp);
    }
}

f2 f2_both(float v) {
    unsigned u;
    memcpy(&u, &v, 4);
    return ((f2)u << 32) | u;
}

template <class Tile, class K>
cudaError_t launch_tiles(SsimArgs &a, bool pixels, K kern, cudaStream_t st) {
    unsigned tiles = 0;
    for (int i = 0; i < a.n; ++i) {
        SsimPlane &p = a.p[i];
        const int h = pixels ? p.h : p.h - 10, w = pixels ? p.w : p.w - 10;
        p.tile0 = tiles;
        p.tiles_x = (unsigned)((w + kTW - 1) / kTW);
        tiles += p.tiles_x * (unsigned)((h + Tile::TH - 1) / Tile::TH);
    }
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Tile::bytes);
    if (e != cudaSuccess) return e;
    kern<<<tiles, kThreads, Tile::bytes, st>>>(a);
    return cudaGetLastError();
}

}  // namespace

// a.p[i]: x, y, pitches, h, w, sum (zeroed), and with `grad` also grad, scale,
// scale_exp, P4 and P2; n <= kRefinePlanes.
cudaError_t launch_ssim(SsimArgs &a, bool grad, int num_sms, cudaStream_t st) {
    double g[11], s = 0.0;
    for (int i = 0; i < 11; ++i) {
        const double r = i - 5.0;
        g[i] = exp(-(r * r) / (2.0 * 1.5 * 1.5));
        s += g[i];
    }
    for (int i = 0; i < 11; ++i) {
        const df v = df_split(g[i] / s);
        a.gh[i] = f2_both(v.hi);
        a.ngh[i] = f2_both(-v.hi);
        a.ngl[i] = f2_both(-v.lo);
    }
    a.c1 = df_split((0.01 * 255.0) * (0.01 * 255.0));
    a.c2 = df_split((0.03 * 255.0) * (0.03 * 255.0));
    // high tiles do least work twice (64 rows for 54); images that would fill
    // less than half of the SMs with them take low ones (32 for 22)
    unsigned high = 0;
    for (int i = 0; i < a.n; ++i)
        high += (unsigned)((a.p[i].w + kTW - 1) / kTW) * (unsigned)((a.p[i].h + 53) / 54);
    const bool low = high * 2 < (unsigned)num_sms;
    cudaError_t e = low ? launch_tiles<FwdTile<3>>(a, false, ssim_forward_kernel<3>, st)
                        : launch_tiles<FwdTile<7>>(a, false, ssim_forward_kernel<7>, st);
    if (e != cudaSuccess || !grad) return e;
    return low ? launch_tiles<BwdTile<4>>(a, true, ssim_backward_kernel<4>, st)
               : launch_tiles<BwdTile<9>>(a, true, ssim_backward_kernel<9>, st);
}

}  // namespace aqmp
