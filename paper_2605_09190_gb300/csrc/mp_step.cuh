// mp_step.cuh -- per-step building blocks shared by the pursuit kernels
// (mp.cu, mp_cluster.cu): step records, summaries of magnitudes and the
// leader's look-up, and the rank-1 correlation update of one atom family.
#pragma once
#include <cuda_runtime.h>

#include "common.cuh"
#include "f32x2.cuh"

namespace aqmp {

struct StepRec {
    uint32_t j;
    float hi, lo;
};

constexpr uint32_t kNone = 0xffffffffu;

// Whether the energy lies within 2^-37 ||y||^2 of the threshold in FP64; out
// of line, so that its FP64 work runs only when the FP32 pre-test asks.
static __device__ __noinline__ bool energy_in_band(df En, df thrE, uint32_t e0) {
    return fabs(df_to_double(En) - df_to_double(thrE)) < ldexp((double)e0, -37);
}

// Top-2 summary of a set of correlations.  P packs the largest |hi| (its
// float bits, high word) with (0xffff - index) << 1 | sign(hi) (low word), so
// the unsigned maximum of P picks the largest magnitude and, among equal
// magnitudes, the lowest index; k2 is the second largest |hi| bits (equal to
// the largest when two atoms share it) and lo1 the low word of the top.
struct Top2 {
    unsigned long long P;
    uint32_t k2;
    float lo1;
};

__device__ __forceinline__ Top2 top2_empty() { return Top2{0ull, 0u, 0.0f}; }

__device__ __forceinline__ unsigned long long top2_key(float hi, uint32_t j) {
    const uint32_t h = __float_as_uint(hi);
    return ((unsigned long long)(h & 0x7fffffffu) << 32) | (((0xffffu - j) << 1) | (h >> 31));
}

// Fold one element into a running top-2.
__device__ __forceinline__ void top2_fold(Top2 &t, float hi, float lo, uint32_t j) {
    const unsigned long long Pe = top2_key(hi, j);
    t.k2 = max(t.k2, min((uint32_t)(t.P >> 32), (uint32_t)(Pe >> 32)));
    const bool take = Pe > t.P;
    t.P = take ? Pe : t.P;
    t.lo1 = take ? lo : t.lo1;
}

__device__ __forceinline__ uint32_t top2_index(const Top2 &t) { return 0xffffu - (((uint32_t)t.P & 0x1ffffu) >> 1); }
__device__ __forceinline__ bool top2_negative(const Top2 &t) { return ((uint32_t)t.P & 1u) != 0u; }
__device__ __forceinline__ float top2_amax(const Top2 &t) { return __uint_as_float((uint32_t)(t.P >> 32)); }

// A thread's E correlations as double-float pairs, slots 2 i and 2 i + 1 of
// the high (low) words in one register pair.
template <int E>
struct Corr {
    f2 h[E / 2], l[E / 2];
    __device__ __forceinline__ float hi(int s) const { return s & 1 ? f2_y(h[s / 2]) : f2_x(h[s / 2]); }
    __device__ __forceinline__ float lo(int s) const { return s & 1 ? f2_y(l[s / 2]) : f2_x(l[s / 2]); }
    __device__ __forceinline__ void set(int s, float vh, float vl) {
        h[s / 2] = s & 1 ? f2_make(f2_x(h[s / 2]), vh) : f2_make(vh, f2_y(h[s / 2]));
        l[s / 2] = s & 1 ? f2_make(f2_x(l[s / 2]), vl) : f2_make(vl, f2_y(l[s / 2]));
    }
};

// Which atoms a thread holds.  A family's b^2 atoms (p, q), index q b + p,
// are spread over VT threads, G slots each: thread v keeps row p = v mod b
// and the G consecutive columns q = G (v / b) + s.  Consecutive columns let
// the rank-1 update read four entries of a W row with one 16-byte load and
// put two of them into one packed FP32 instruction; a thread's atom index
// still grows with the slot.  A thread that holds both families has slots
// [0, G) in the first and [G, 2 G) in the second.
template <int B, int VT, int G>
struct Atoms {
    static constexpr uint32_t n = B * B;
    static_assert(G * VT == B * B && VT % B == 0, "layout");
    // atom of thread v's slot 0 in its (first) family `fam`
    static __device__ __forceinline__ uint32_t base(int v, int fam) {
        return (uint32_t)fam * n + (uint32_t)(v % B) + (uint32_t)(B * G) * (uint32_t)(v / B);
    }
    // atom of slot s given the base
    static __device__ __forceinline__ uint32_t atom(uint32_t base, int s) {
        return base + (uint32_t)(s / G) * n + (uint32_t)B * (uint32_t)(s % G);
    }
    // the thread of the family that holds atom j, and its slot there
    static __device__ __forceinline__ uint32_t owner(uint32_t j) {
        const uint32_t f = j % n;
        return f % B + (uint32_t)B * (f / (uint32_t)(B * G));
    }
    static __device__ __forceinline__ uint32_t slot(uint32_t j) { return (j % n) / B % G; }
};

__device__ __forceinline__ float max3(float a, float b, float c) {
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

__device__ __forceinline__ float max3_abs(float a, float b, float c) {
    float d;
    asm("max.abs.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

// A thread's per-step summary: the largest magnitude of each group of up to
// eight slots (of one family).  It costs half an instruction an element; the
// ALU work of carrying sign, slot, low word and runner-up along would take
// half as long again as the update itself, since it shares the issue slots
// with the packed FP32 instructions.  Those words are looked up once a step,
// by the one warp that holds the leader.
template <int E, int G>
struct Summary {
    static constexpr int GS = G < 8 ? G : 8, N = E / GS;
    float g[N];
    __device__ __forceinline__ float top() const {
        float m = g[0];
#pragma unroll
        for (int i = 1; i < N; ++i) m = fmaxf(m, g[i]);
        return m;
    }
    // slots [S0, S0 + GN) as they stand
    template <int S0, int GN>
    __device__ __forceinline__ void form(const Corr<E> &c) {
#pragma unroll
        for (int i = S0 / GS; i < (S0 + GN) / GS; ++i) {
            g[i] = 0.0f;
#pragma unroll
            for (int s = i * GS; s < (i + 1) * GS; s += 2) g[i] = max3_abs(g[i], c.hi(s), c.hi(s + 1));
        }
    }
};

struct Pair2 {
    float m1, m2;
};

__device__ __forceinline__ void fold2(Pair2 &k, float a, float b) {
    const float mx = fmaxf(a, b);
    k.m2 = max3(k.m2, fminf(a, b), fminf(k.m1, mx));
    k.m1 = fmaxf(k.m1, mx);
}

// The two largest magnitudes themselves, of all E slots.
template <int E>
__device__ __forceinline__ Pair2 magnitudes_of(const Corr<E> &c) {
    Pair2 k{0.0f, 0.0f};
#pragma unroll
    for (int s = 0; s < E; s += 2) fold2(k, fabsf(c.hi(s)), fabsf(c.hi(s + 1)));
    return k;
}

// The words of slot S0 + s (0 <= s < N); straight-line.
template <int E, int N, int S0>
__device__ __forceinline__ df pick_slot(const Corr<E> &c, uint32_t s) {
    if constexpr (N == 1) {
        return df{c.hi(S0), c.lo(S0)};
    } else {
        const df a = pick_slot<E, N / 2, S0>(c, s), b = pick_slot<E, N / 2, S0 + N / 2>(c, s);
        const bool up = (s & (uint32_t)(N / 2)) != 0u;
        return df{up ? b.hi : a.hi, up ? b.lo : a.lo};
    }
}

// The leader of a warp or of a group: its words, its atom, and the largest of
// all other magnitudes (float bits).  Where that equals |hi| (two atoms share
// the largest magnitude) the words and the atom may be no one atom's.
struct Lead {
    float hi, lo;
    uint32_t j, k2;
};

__device__ __forceinline__ Lead unpack_lead(const uint4 &v) {
    return Lead{__uint_as_float(v.x), __uint_as_float(v.y), v.z, v.w};
}

// The largest M of the warp's k1 and the lanes that hold it, and the second:
// the largest of the holder's own second `second` and the other lanes' k1, or
// M again where two lanes hold it.
__device__ __forceinline__ void warp_two(uint32_t k1, uint32_t second, uint32_t &M, uint32_t &M2, bool &holds) {
    M = __reduce_max_sync(0xffffffffu, k1);
    holds = k1 == M;
    const uint32_t others = __reduce_max_sync(0xffffffffu, holds ? second : k1);
    M2 = __reduce_add_sync(0xffffffffu, holds ? 1u : 0u) > 1u ? M : others;
}

// Looks a group of slots over for the magnitude M: its words and slot, and
// the largest of the others (M where two share it).
template <int E, int GS, int S0>
__device__ __forceinline__ void look_over(const Corr<E> &c, uint32_t M, df &w, uint32_t &slot, uint32_t &second) {
    const float Mf = __uint_as_float(M);
    uint32_t found = 0u;
    float rest[GS];
#pragma unroll
    for (int i = 0; i < GS; ++i) {
        const float h = c.hi(S0 + i);
        const bool is = fabsf(h) == Mf;
        w.hi = is ? h : w.hi;
        w.lo = is ? c.lo(S0 + i) : w.lo;
        slot = is ? (uint32_t)(S0 + i) : slot;
        found |= is ? 1u << i : 0u;
        rest[i] = is ? 0.0f : fabsf(h);
    }
#pragma unroll
    for (int i = 2; i < GS; i += 2) rest[i % 4 / 2] = max3(rest[i % 4 / 2], rest[i], rest[i + 1]);
    second = (found & (found - 1u)) != 0u ? M : __float_as_uint(fmaxf(rest[0], rest[1]));
}

template <int E, int G, int I, int N>
__device__ __forceinline__ void look_in_group(const Corr<E> &c, int i, uint32_t M, df &w, uint32_t &slot,
                                              uint32_t &second) {
    if constexpr (N == 1) {
        look_over<E, Summary<E, G>::GS, I * Summary<E, G>::GS>(c, M, w, slot, second);
    } else {
        if (i & (N / 2)) look_in_group<E, G, I + N / 2, N / 2>(c, i, M, w, slot, second);
        else look_in_group<E, G, I, N / 2>(c, i, M, w, slot, second);
    }
}

// The warp that holds the largest magnitude M on the lane with `holds` set:
// that lane writes the leader, with its own second magnitude, to *dst.
template <class At, int E, int G>
__device__ __forceinline__ void write_lead(const Summary<E, G> &sm, const Corr<E> &c, uint32_t base, uint32_t M,
                                           bool holds, uint32_t second, uint4 *dst) {
    constexpr int N = Summary<E, G>::N;
    uint32_t in = 0u, rest = 0u;               // the groups that reach M, the largest of the others
#pragma unroll
    for (int i = 0; i < N; ++i) {
        const uint32_t v = __float_as_uint(sm.g[i]);
        if (v == M) in |= 1u << i;
        else rest = max(rest, v);
    }
    // one of the lane's groups (several: the caller decides); uniform
    const uint32_t groups = N == 1 ? 1u : __reduce_or_sync(0xffffffffu, holds ? in : 0u);
    df w{0.0f, 0.0f};
    uint32_t slot = 0u, sec = 0u;
    look_in_group<E, G, 0, N>(c, 31 - __clz((int)groups), M, w, slot, sec);
    // (the magnitude is M whatever was found: two lanes may hold it in
    // different groups, and only one group was looked over)
    if (holds)
        *dst = make_uint4((__float_as_uint(w.hi) & 0x80000000u) | M, __float_as_uint(w.lo), At::atom(base, (int)slot),
                          (in & (in - 1u)) != 0u ? M : max(max(sec, rest), second));
}

__device__ __forceinline__ void warp_argmax64(unsigned long long &bk, uint32_t &bj) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const unsigned long long ok = __shfl_xor_sync(0xffffffffu, bk, off);
        const uint32_t oj = __shfl_xor_sync(0xffffffffu, bj, off);
        if (ok > bk || (ok == bk && oj < bj)) {
            bk = ok;
            bj = oj;
        }
    }
}

__device__ __forceinline__ uint32_t warp_min(uint32_t v) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v = min(v, __shfl_xor_sync(0xffffffffu, v, off));
    return v;
}

// c - u w for two correlations at once with the packed FP32 instructions
// (two independent IEEE operations each): df_sub_mul operation for
// operation, so each half has its bits.  uh, nuh, ul hold u.hi, -u.hi, u.lo
// twice; a - b is formed as fma(b, -1, a), which rounds the same.
__device__ __forceinline__ void df_sub_mul2(f2 &ch, f2 &cl, f2 uh, f2 nuh, f2 ul, f2 m1, f2 wh, f2 wl) {
    const f2 np = f2_mul(nuh, wh);                              // -(u.hi w.hi), rounded
    const f2 pe = f2_fma(ul, wh, f2_fma(uh, wl, f2_fma(uh, wh, np)));
    const f2 s = f2_add(ch, np);
    const f2 bb = f2_fma(ch, m1, s);
    const f2 x = f2_fma(f2_fma(bb, m1, s), m1, ch);
    const f2 y = f2_fma(bb, m1, np);
    const f2 e = f2_add(f2_add(x, y), f2_fma(pe, m1, cl));
    ch = f2_add(s, e);
    cl = f2_fma(f2_fma(s, m1, ch), m1, e);
}

// Rank-1 update of the elements in slots [S0, S0 + G) (one atom family) and
// their part of the summary.  whi and wlo point at this thread's G consecutive
// columns of row q* of the W table's two planes (high and low words): every
// lane of a row group reads the same 16 bytes.
//
// 15 operations per element, in 7.5 packed instructions of two issue slots
// each.  At the FP32 rate that is 2.4 of the 7.9 ms of 50 910 leaves of side 64
// (1.58 M steps); the rest of a step is its exchange and look-up (mp.cu).
template <int E, int G, int S0, bool DF>
__device__ __forceinline__ void update_family(Corr<E> &c, Summary<E, G> &sm, const df &u, const float *whi,
                                              const float *wlo) {
    constexpr int GS = Summary<E, G>::GS;
    static_assert(G % 2 == 0, "pairs of slots");
    constexpr int W = G % 4 == 0 ? 2 : 1;                        // column pairs per load
    const f2 uh = f2_make(u.hi, u.hi), nuh = f2_make(-u.hi, -u.hi), ul = f2_make(u.lo, u.lo);
    const f2 m1 = f2_make(-1.0f, -1.0f);
#pragma unroll
    for (int i = 0; i < G / GS; ++i) sm.g[S0 / GS + i] = 0.0f;
#pragma unroll
    for (int s2 = 0; s2 < G; s2 += 2 * W) {
        f2 wh[W], wl[W];
        if constexpr (W == 2) {
            const ulonglong2 h = *reinterpret_cast<const ulonglong2 *>(whi + s2);
            wh[0] = h.x;
            wh[1] = h.y;
            if (DF) {
                const ulonglong2 l = *reinterpret_cast<const ulonglong2 *>(wlo + s2);
                wl[0] = l.x;
                wl[1] = l.y;
            }
        } else {
            wh[0] = *reinterpret_cast<const f2 *>(whi + s2);
            if (DF) wl[0] = *reinterpret_cast<const f2 *>(wlo + s2);
        }
#pragma unroll
        for (int i = 0; i < W; ++i) {
            const int s = S0 + s2 + 2 * i;
            if (DF) df_sub_mul2(c.h[s / 2], c.l[s / 2], uh, nuh, ul, m1, wh[i], wl[i]);
            else c.h[s / 2] = f2_fma(nuh, wh[i], c.h[s / 2]);     // plain FP32 form: one FMA per entry
            sm.g[s / GS] = max3_abs(sm.g[s / GS], c.hi(s), c.hi(s + 1));
        }
    }
}

// Zero slot S0 + s2 (none if s2 is not in [0, G)); straight-line, the
// registers stay statically indexed.
template <int E, int G, int S0>
__device__ __forceinline__ void zero_slot(Corr<E> &c, int s2) {
#pragma unroll
    for (int i = 0; i < G; ++i)
        if (i == s2) c.set(S0 + i, 0.0f, 0.0f);
}

}  // namespace aqmp
