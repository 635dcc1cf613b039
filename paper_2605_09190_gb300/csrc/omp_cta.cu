// omp_cta.cu -- Orthogonal Matching Pursuit per leaf (the solver the paper's
// authors ran, Section 2.2) at sides 32 and 64, with the quadtree split /
// emit of Algorithm 2.  The rules are those of omp.cu (sides 4..16): the
// residual energy ||y||^2 - |z|^2 tested before each step (Eq. (3), strict,
// with the MP kernel's equality band), the residual correlations
// c = c0 - G[:, S] x_S outside the support, argmax |c| with ties within
// 2^-32 ||y|| going to the lowest index, the inverse factor K = L^-1 of G_SS
// grown by a row per selection (a pivot <= 2^-40 ends the pursuit), and the
// re-fit x_S += z_new times that row.  Everything is FP64, at 1/64 of GB300's
// FP32 rate: FP64 instructions bound a leaf in flight (16 SM cycles a warp), so the
// work is cut by structure and spread over idle SMs.
//
// A cluster of C CTAs owns one leaf (as many as the level's leaves leave SMs
// for).  CTA r holds the correlations of the atoms (p, q) with q in its b / C
// columns, of both families.
//
// Cross terms.  The Gram matrix is the identity inside a family and
// kron(W, W) across (W = C H^T), so the DCT atoms need W U with
// U = X_H W^T restricted to the CTA's columns, and the Haar atoms W^T V with
// V = X_C W (X_F the family's coefficients as a b x b matrix).  U and V are
// formed from the support lists, row by row (a few terms per entry).  The
// remaining product is halved by mirror symmetry: with h' the mirror image of
// Haar row h at its scale, W[p][h'] = -(-1)^p W[p][h], so with D = U[h] - U[h']
// and S = U[h] + U[h'] an even p takes W[p][h] D and an odd p W[p][h] S over
// one h of each pair; and (W^T V)[h], [h'] = +-A + O with A, O the sums over
// even and odd p.  32 terms for two entries, against 64 each for the dense
// product that was formed in two full b x b x b steps before.
//
// Factor.  K lives in a global slot per cluster twice, by rows and by columns,
// so that K g (a thread per row; g is zero on the new atom's own family) and
// w^T K (a thread per column) both read contiguously; each CTA takes a share
// of the rows and of the columns and the results meet through distributed
// shared memory: three cluster barriers a step.  Every sum is formed in an order
// that the support alone fixes, so the coefficients have the same bits at every
// width of the cluster.
// Piecewise scenes, whole encodes against one CTA a leaf with dense cross terms
// and triangular solves: 256x256 of 64x64 roots 115 -> 10.5 ms, 512x512 67.2 ->
// 19.8, 1024x640 (160 leaves, one CTA each) 42.0 -> 24.0; 512x512 of 32x32 roots
// 26.1 -> 13.1; 512x512 at four tolerances down to side 4, up to 1024 atoms a
// leaf, 883 -> 546.
#include <cuda_runtime.h>

#include "common.cuh"
#include "kernels.h"

namespace aqmp {

namespace {

constexpr double kTieRel = 0x1p-32;
constexpr double kBandRel = 0x1p-37;
constexpr double kPivotMin = 0x1p-40;
constexpr uint32_t kNoAtom = 0xffffffffu;
constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kMaxBudget = 1024;

__host__ __device__ __forceinline__ long long tri64(long long i) { return i * (i + 1) / 2; }
// Doubles of a slot: K by rows and by columns, both packed.
__host__ __device__ __forceinline__ long long slot_doubles(long long k) { return 2 * tri64(k); }
// Where row 0 of column c of K would be in the packed columns (its rows are c .. k - 1).
__device__ __forceinline__ int column_at(int c, int k) { return c * (2 * k - c - 1) / 2; }

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    return v;
}

// |v| as an integer of the same order.
__device__ __forceinline__ unsigned long long mag_bits(double v) {
    return (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
}

__device__ __forceinline__ unsigned long long warp_max64(unsigned long long v) {
    const uint32_t hi = __reduce_max_sync(0xffffffffu, (uint32_t)(v >> 32));
    const uint32_t lo = __reduce_max_sync(0xffffffffu, (uint32_t)(v >> 32) == hi ? (uint32_t)v : 0u);
    return ((unsigned long long)hi << 32) | lo;
}

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

__device__ __forceinline__ uint32_t cluster_id() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%clusterid.x;" : "=r"(r));
    return r;
}

// All threads of the cluster; writes before it (shared memory of any CTA of
// the cluster, global memory) are seen after it.
template <int C>
__device__ __forceinline__ void cluster_sync() {
    if (C == 1) __syncthreads();
    else asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Writes v to the same shared-memory variable of CTA `rank`.
__device__ __forceinline__ void put(double *p, uint32_t rank, double v) {
    uint32_t at;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(at) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(at), "d"(v) : "memory");
}

// ... of every CTA of the cluster.
template <int C>
__device__ __forceinline__ void put_all(double *p, double v) {
    if (C == 1) {
        *p = v;
        return;
    }
#pragma unroll
    for (uint32_t r = 0; r < (uint32_t)C; ++r) put(p, r, v);
}

// How many partial sums a row's or a column's product with the factor is formed
// as, given the 32-row blocks of the support: by its size alone, and joined as
// a tree over neighbours, so that a leaf's coefficients have the same bits
// whatever the cluster's width (how many leaves share the call, which GPU runs
// it).  As many as the warps a block gets at the widest cluster.
constexpr int kMaxBlocks = kMaxBudget / 32;
__device__ __forceinline__ int parts_of(int blocks) { return blocks <= 8 ? 8 : blocks <= 16 ? 4 : 2; }
static_assert(kWarps == 8 && kMaxBlocks <= 32, "partial sums, one block a lane");

// p[0] .. p[(n - 1) stride], n a power of two up to 8, joined as that tree.
__device__ __forceinline__ double join_tree(const double *p, int stride, int n) {
    double v = p[0];
    if (n >= 2) v += p[stride];
    if (n >= 4) v += p[2 * stride] + p[3 * stride];
    if (n >= 8) v += (p[4 * stride] + p[5 * stride]) + (p[6 * stride] + p[7 * stride]);
    return v;
}

// Partial sums at, at + 1 .. at + m - 1 of `of` (a power of two; m one too) of
// the terms first .. count - 1, partial s taking first + s, first + s + of ...,
// joined: term(i, sum) adds term i.
template <int MP, class Term>
__device__ __forceinline__ double partial_sums_n(int first, int count, int at, int of, Term term) {
    double p[MP];
#pragma unroll
    for (int e = 0; e < MP; ++e) p[e] = 0.0;
#pragma unroll(MP >= 4 ? 1 : 4 / MP)
    for (int i = first + at; i < count; i += of) {
#pragma unroll
        for (int e = 0; e < MP; ++e)
            if (i + e < count) p[e] = term(i + e, p[e]);
    }
#pragma unroll
    for (int w = 1; w < MP; w *= 2)
#pragma unroll
        for (int e = 0; e + w < MP; e += 2 * w) p[e] += p[e + w];
    return p[0];
}

template <class Term>
__device__ __forceinline__ double partial_sums(int first, int count, int at, int m, int of, Term term) {
    if (m == 1) return partial_sums_n<1>(first, count, at, of, term);
    if (m == 2) return partial_sums_n<2>(first, count, at, of, term);
    if (m == 4) return partial_sums_n<4>(first, count, at, of, term);
    return partial_sums_n<8>(first, count, at, of, term);
}

// What one CTA offers to the step's choice.
struct Offer {
    double amax;               // its largest |c|
    double c0;                 // of the atom below
    double j;                  // lowest index within the tie window of amax
    double tie;                // (CTA 0's copy) whether a decision fell into a certification band
};

// Shared-memory layout.
template <int B, int NF, int C>
struct OmpLayout {
    static constexpr int n = B * B, M = NF * n;
    static constexpr int Q = B / C;                 // columns of a CTA
    static constexpr int NP = B / 2;                // pairs of rows
    static constexpr int CT = kThreads / NP;        // columns the threads take at a time
    static constexpr int EQ = (Q + CT - 1) / CT;    // columns per thread
    static constexpr int SUB = kThreads / B;        // threads per row when U and V are formed
    static constexpr int ES = Q / SUB;              // columns per such thread
    static_assert(Q % SUB == 0 && ES >= 1, "columns");
    // doubles: WP[p][i] and its transpose (pairs), the column slices of W and
    // W^T, V and U, then per-support arrays
    static constexpr int wp = 0, wpt = wp + (NF == 2 ? B * NP : 0), wq = wpt + (NF == 2 ? B * NP : 0),
                         wtq = wq + (NF == 2 ? B * Q : 0), vv = wtq + (NF == 2 ? B * Q : 0),
                         uu = vv + (NF == 2 ? B * Q : 0), red = uu + (NF == 2 ? B * Q : 0),
                         offers = red + 2 * kWarps, sums = offers + 4 * C, claim = sums + 2 * kMaxBlocks, part = claim + 2,
                         arrays = part + kThreads;
    __host__ __device__ static constexpr size_t doubles(int k) { return (size_t)arrays + 4 * (size_t)k; }
    // words: the support's atoms, their predecessors in their row, the positions by family; row heads; misc
    __host__ __device__ static constexpr size_t bytes(int k) {
        return 8 * doubles(k) + 4 * (3 * (size_t)k + 2 * B + 16);
    }
};

// The Haar row of pair i (the other is mirror(h)); pair B / 2 - 1 stands for
// rows 0 and 1.  Pair i at scale s = 2^(1 + floor(log2(i + 1))): h = i + 1 + s / 2.
__host__ __device__ __forceinline__ int pair_row(int i, int np) {
    if (i == np - 1) return 1;
    int half = 1;
    while (2 * half <= i + 1) half *= 2;
    return i + 1 + half;
}
__host__ __device__ __forceinline__ int mirror_row(int h) {
    int s = 1;
    while (2 * s <= h) s *= 2;
    return 3 * s - 1 - h;
}

}  // namespace

template <int B, int NF, int C>
__global__ void __launch_bounds__(kThreads, 1) omp_cta_kernel(MPArgs a) {
    using Ly = OmpLayout<B, NF, C>;
    constexpr int n = Ly::n, M = Ly::M, Q = Ly::Q, NP = Ly::NP, CT = Ly::CT, EQ = Ly::EQ;

    extern __shared__ __align__(16) double sm[];
    double *WP = sm + Ly::wp, *WPT = sm + Ly::wpt;     // W[p][h_i]: [p][i], [i][p]
    double *WQ = sm + Ly::wq, *WTQ = sm + Ly::wtq;     // W[q'][q] and W[q][q'], q of this CTA: [q'][q]
    double *V = sm + Ly::vv, *U = sm + Ly::uu;         // [row][q]
    double *red = sm + Ly::red;
    Offer *offers = reinterpret_cast<Offer *>(sm + Ly::offers);
    double *sums = sm + Ly::sums;                      // [block of 32 rows][2]: |w|^2 and w . z
    double *part = sm + Ly::part;
    const int k = a.lv.k;
    double *xs = sm + Ly::arrays, *zs = xs + k, *gs = zs + k, *wv = gs + k;
    uint32_t *Sj = reinterpret_cast<uint32_t *>(wv + k);
    uint32_t *prev = Sj + k;                           // the atom before in the same row and family
    uint32_t *fam_pos = prev + k;                      // positions of the DCT atoms, from the end the Haar atoms
    uint32_t *head = fam_pos + k;                      // [2][B] last atom of each row p
    uint32_t *bc = head + 2 * B;                       // broadcast words

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rank = C == 1 ? 0 : (int)cluster_rank();
    const int cid = C == 1 ? (int)blockIdx.x : (int)cluster_id();
    const int q0 = rank * Q;
    if (NF == 2) {
        auto w_at = [&](int p, int h) { const float2 w = a.W[p * B + h]; return (double)w.x + (double)w.y; };
        for (int i = tid; i < B * NP; i += kThreads) {
            const double w = w_at(i / NP, pair_row(i % NP, NP));
            WP[i] = w;
            WPT[(i % NP) * B + i / NP] = w;
        }
        for (int i = tid; i < B * Q; i += kThreads) {
            WQ[i] = w_at(i / Q, q0 + i % Q);
            WTQ[i] = w_at(q0 + i % Q, i / Q);
        }
    }
    // this thread's pair of rows and columns
    const int pr = tid % NP, qc = tid / NP;
    const int hp = pair_row(pr, NP), hm = pr == NP - 1 ? 0 : mirror_row(hp);
    cluster_sync<C>();

    const LevelArgs &lv = a.lv;
    const unsigned count = *lv.count;
    double *Kr = a.omp_L + (size_t)cid * (size_t)slot_doubles(k), *Kc = Kr + tri64(k);
    unsigned *work = &a.ctr->work_next[lv.level];
    double *claim = sm + Ly::claim;

    for (;;) {
        // dynamic assignment: CTA 0 of the cluster takes the next unclaimed leaf
        if (rank == 0 && tid == 0) put_all<C>(claim, (double)atomicAdd(work, 1u));
        cluster_sync<C>();
        const double claimed = *claim;
        __syncthreads();
        if (claimed >= (double)count) break;
        const unsigned leaf = (unsigned)claimed;

        const QueueEntry qe = lv.queue[leaf];
        const double tol = (double)a.planes[qe.plane].tol;
        const double eps2 = tol * tol * (double)n;
        const double E0 = (double)a.e0[leaf];
        const double Sy = sqrt(E0);
        const double tie_c = kTieRel * Sy, band_c = kBandRel * Sy;
        const double thr_e = eps2 - kTieRel * E0, band_e = kBandRel * E0;

        // entries: DCT rows 2 pr and 2 pr + 1, Haar rows hp and hm; index
        // 4 e + {0, 1, 2, 3} for column qc + CT e
        double c0r[4 * EQ];
        const float2 *cp = a.c0 + (size_t)leaf * M;
        auto atom_of = [&](int i) {
            const int q = q0 + qc + CT * (i / 4), f = i % 4;
            const int p = NF == 1 || f < 2 ? 2 * pr + f : f == 2 ? hp : hm;
            return (uint32_t)(q * B + p + (f >= 2 ? n : 0));
        };
        auto is_here = [&](int i) { return (NF == 2 || i % 4 < 2) && qc + CT * (i / 4) < Q; };
#pragma unroll
        for (int i = 0; i < 4 * EQ; ++i) {
            c0r[i] = 0.0;
            if (is_here(i)) {
                const float2 v = cp[atom_of(i)];
                c0r[i] = (double)v.x + (double)v.y;
            }
        }
        for (int i = tid; i < 2 * B; i += kThreads) head[i] = kNoAtom;
        __syncthreads();
        uint32_t taken = 0u;
        int nS = 0, nC = 0, nH = 0;          // support size, and per family
        double En = E0;                       // alike on every thread of the cluster
        bool conv = false, tie = false;
        for (;;) {
            // (a6) accuracy test before every step, strict
            if (fabs(En - thr_e) < band_e) tie = true;
            if (En < thr_e) { conv = true; break; }
            if (nS == k) break;

            double cv[4 * EQ];
#pragma unroll
            for (int i = 0; i < 4 * EQ; ++i) cv[i] = c0r[i];
            if (NF == 2 && nS > 0) {
                // U[a][q] = sum x W[q][b] over the Haar atoms (a, b), and
                // V[p][q] = sum x W[b][q] over the DCT atoms (p, b)
                const int row = tid / Ly::SUB, c = tid % Ly::SUB;
                double u[Ly::ES], v[Ly::ES];
#pragma unroll
                for (int e = 0; e < Ly::ES; ++e) u[e] = v[e] = 0.0;
                for (uint32_t i = head[B + row]; i != kNoAtom; i = prev[i]) {
                    const double x = xs[i];
                    const double *w = WTQ + (Sj[i] - (uint32_t)n) / B * Q + c;
#pragma unroll
                    for (int e = 0; e < Ly::ES; ++e) u[e] = fma(x, w[Ly::SUB * e], u[e]);
                }
                for (uint32_t i = head[row]; i != kNoAtom; i = prev[i]) {
                    const double x = xs[i];
                    const double *w = WQ + Sj[i] / B * Q + c;
#pragma unroll
                    for (int e = 0; e < Ly::ES; ++e) v[e] = fma(x, w[Ly::SUB * e], v[e]);
                }
#pragma unroll
                for (int e = 0; e < Ly::ES; ++e) {
                    U[row * Q + c + Ly::SUB * e] = u[e];
                    V[row * Q + c + Ly::SUB * e] = v[e];
                }
                __syncthreads();
                // rows h and h' of a pair become D and S (rows 0 and 1 stay)
                for (int i = tid; i < (NP - 1) * Q; i += kThreads) {
                    const int h = pair_row(i / Q, NP), q = i % Q;
                    double *uh = U + h * Q + q, *um = U + mirror_row(h) * Q + q;
                    const double x = *uh, y = *um;
                    *uh = x - y;
                    *um = x + y;
                }
                __syncthreads();
                double s0[EQ], s1[EQ], sa[EQ], so[EQ];
#pragma unroll
                for (int e = 0; e < EQ; ++e) s0[e] = s1[e] = sa[e] = so[e] = 0.0;
                if (nH > 0) {
                    for (int half = 1; half < NP; half *= 2)
#pragma unroll 4
                        for (int t = 0; t < half; ++t) {
                            const double2 w = *reinterpret_cast<const double2 *>(WPT + (half - 1 + t) * B + 2 * pr);
                            const double *ud = U + (2 * half + t) * Q, *us = U + (4 * half - 1 - t) * Q;
#pragma unroll
                            for (int e = 0; e < EQ; ++e) {
                                const int q = min(qc + CT * e, Q - 1);
                                s0[e] = fma(w.x, ud[q], s0[e]);
                                s1[e] = fma(w.y, us[q], s1[e]);
                            }
                        }
                    // row 1 is its own mirror image: the odd p alone
                    const double w = WPT[(NP - 1) * B + 2 * pr + 1];
#pragma unroll
                    for (int e = 0; e < EQ; ++e) s1[e] = fma(w, U[Q + min(qc + CT * e, Q - 1)], s1[e]);
                }
                if (nC > 0) {
#pragma unroll 4
                    for (int p = 0; p < B; p += 2) {
                        const double we = WP[p * NP + pr], wo = WP[(p + 1) * NP + pr];
#pragma unroll
                        for (int e = 0; e < EQ; ++e) {
                            const int q = min(qc + CT * e, Q - 1);
                            sa[e] = fma(we, V[p * Q + q], sa[e]);
                            so[e] = fma(wo, V[(p + 1) * Q + q], so[e]);
                        }
                    }
                }
#pragma unroll
                for (int e = 0; e < EQ; ++e) {
                    const int q = min(qc + CT * e, Q - 1);
                    cv[4 * e] -= s0[e] + (pr == 0 ? U[q] : 0.0);
                    cv[4 * e + 1] -= s1[e];
                    // rows 0 and 1: W[p][0] is 1 at p = 0 alone
                    cv[4 * e + 2] -= pr == NP - 1 ? so[e] : sa[e] + so[e];
                    cv[4 * e + 3] -= pr == NP - 1 ? V[q] : so[e] - sa[e];
                }
            }
            // this CTA's largest, and its lowest index within the tie window
            unsigned long long mag[4 * EQ], best = 0ull;
#pragma unroll
            for (int i = 0; i < 4 * EQ; ++i) {
                mag[i] = is_here(i) && !((taken >> i) & 1u) ? mag_bits(cv[i]) : 0ull;
                best = max(best, mag[i]);
            }
            best = warp_max64(best);
            if (lane == 0) red[warp] = __longlong_as_double((long long)best);
            __syncthreads();
            double mine = red[0];
#pragma unroll
            for (int w = 1; w < kWarps; ++w) mine = fmax(mine, red[w]);
            // the lowest index with |c| >= edge, and its c0, to offers[rank] of
            // every CTA; whether any value lies within a band of the edge
            auto offer = [&](double edge) {
                const unsigned long long edge_b = mag_bits(edge);
                const unsigned long long lo = mag_bits(fmax(edge - 2.0 * band_c, 0.0)), hi = mag_bits(edge + 2.0 * band_c);
                uint32_t jl = kNoAtom;
                bool near = false;
#pragma unroll
                for (int i = 0; i < 4 * EQ; ++i) {
                    if (!is_here(i)) continue;
                    if (edge > 0.0 && mag[i] >= edge_b) jl = min(jl, atom_of(i));
                    near |= mag[i] >= lo && mag[i] <= hi;
                }
                bool hit = false;
                if (__builtin_expect(near, 0)) {
#pragma unroll
                    for (int i = 0; i < 4 * EQ; ++i)
                        if (is_here(i) && fabs(__longlong_as_double((long long)mag[i]) - edge) < band_c) hit = true;
                }
                const uint32_t jw = __reduce_min_sync(0xffffffffu, jl);
                if (lane == 0) bc[4 + warp] = jw;
                __syncthreads();
                uint32_t jm = bc[4];
#pragma unroll
                for (int w = 1; w < kWarps; ++w) jm = min(jm, bc[4 + w]);
#pragma unroll
                for (int i = 0; i < 4 * EQ; ++i)
                    if (is_here(i) && jm != kNoAtom && atom_of(i) == jm) {
                        put_all<C>(&offers[rank].amax, mine);
                        put_all<C>(&offers[rank].c0, c0r[i]);
                        put_all<C>(&offers[rank].j, (double)jm);
                    }
                if (jm == kNoAtom && tid == 0) {
                    put_all<C>(&offers[rank].amax, mine);
                    put_all<C>(&offers[rank].j, (double)kNoAtom);
                }
                cluster_sync<C>();
                return hit;
            };
            const double my_edge = mine - tie_c;
            bool hit = offer(my_edge);
            double amax = 0.0;
#pragma unroll
            for (int r = 0; r < C; ++r) amax = fmax(amax, offers[r].amax);
            if (amax <= tie_c) break;                        // nothing left to remove
            const double edge = amax - tie_c;
            if (C > 1) {
                // another CTA's largest within reach of the edge: all of them
                // look again at the common edge (else the leader's own is it)
                int reach = 0;
#pragma unroll
                for (int r = 0; r < C; ++r) reach += offers[r].amax >= edge - 4.0 * band_c ? 1 : 0;
                if (reach > 1) {
                    cluster_sync<C>();
                    hit = offer(edge);
                } else if (mine != amax) {
                    hit = false;
                }
            }
            tie |= hit;
            uint32_t jb = kNoAtom;
            double c0b = 0.0;
#pragma unroll
            for (int r = 0; r < C; ++r) {
                const uint32_t j = offers[r].amax >= edge ? (uint32_t)offers[r].j : kNoAtom;
                if (j < jb) {
                    jb = j;
                    c0b = offers[r].c0;
                }
            }
            const bool haar = NF == 2 && jb >= (uint32_t)n;

            // w = K g, g = G[S, jb] (nonzero on the other family alone): rows
            // in blocks of 32 lanes, block b of CTA b mod C, the columns split
            // over the warps that share the block
            double ww = 0.0, wz = 0.0;
            if (NF == 2 && nS > 0) {
                for (int i = tid; i < nS; i += kThreads) {
                    const uint32_t s = Sj[i];
                    double g = 0.0;
                    if ((s >= (uint32_t)n) != haar) {
                        const uint32_t dd = haar ? s : jb, hh = (haar ? jb : s) - (uint32_t)n;
                        const float2 x = a.W[(dd % B) * B + hh % B], y = a.W[(dd / B) * B + hh / B];
                        g = ((double)x.x + (double)x.y) * ((double)y.x + (double)y.y);
                    }
                    gs[i] = g;
                }
                __syncthreads();
                const int others = haar ? nC : nH;
                const int blocks = (nS + 31) / 32, own = (blocks - rank + C - 1) / C;     // blocks of this CTA
                const int parts = parts_of(blocks);
                for (int b0 = 0; b0 < own; b0 += kWarps) {
                    const int nb = min(kWarps, own - b0);
                    const int split = min(parts, nb == 1 ? 8 : nb == 2 ? 4 : nb <= 4 ? 2 : 1);   // warps per block
                    const int ib = warp % nb, is = warp / nb, block = (b0 + ib) * C + rank;
                    const int r = block * 32 + lane;
                    double w = 0.0;
                    if (is < split)
                        w = partial_sums(0, others, is * (parts / split), parts / split, parts, [&](int i, double v) {
                            const int at = (int)fam_pos[haar ? i : k - 1 - i];
                            return r >= at && r < nS ? fma(__ldcg(Kc + column_at(at, k) + r), gs[at], v) : v;
                        });
                    part[tid] = w;
                    __syncthreads();
                    if (is == 0) {
                        w = join_tree(part + ib * 32 + lane, nb * 32, split);
                        if (r < nS) put_all<C>(wv + r, w);
                        ww = warp_sum(w * w);
                        wz = warp_sum(r < nS ? w * zs[r] : 0.0);
                        if (lane == 0) {
                            put_all<C>(sums + 2 * block, ww);
                            put_all<C>(sums + 2 * block + 1, wz);
                        }
                    }
                    __syncthreads();
                }
                cluster_sync<C>();
                // a block a lane: the same tree on every warp of the cluster
                ww = warp_sum(lane < blocks ? sums[2 * lane] : 0.0);
                wz = warp_sum(lane < blocks ? sums[2 * lane + 1] : 0.0);
            }
            const double d = 1.0 - ww;
            if (d > kPivotMin * 0x1p-4 && d < kPivotMin * 0x1p4) tie = true;
            if (d <= kPivotMin) break;                       // dependent on the support
            const double rd = 1.0 / sqrt(d), zn = (c0b - wz) * rd;
            En -= zn * zn;

            // K's new row v = (-w^T K, 1) / sqrt(d) and x_S += zn v: columns in
            // blocks of 32 lanes as the rows above
            {
                const int cols = nS + 1, blocks = (cols + 31) / 32, own = (blocks - rank + C - 1) / C;
                const int parts = parts_of(blocks);
                for (int b0 = 0; b0 < own; b0 += kWarps) {
                    const int nb = min(kWarps, own - b0);
                    const int split = min(parts, nb == 1 ? 8 : nb == 2 ? 4 : nb <= 4 ? 2 : 1);
                    const int ib = warp % nb, is = warp / nb, first = ((b0 + ib) * C + rank) * 32;
                    const int c = first + lane;
                    double v = 0.0;
                    if (NF == 2 && is < split)
                        v = partial_sums(first, nS, is * (parts / split), parts / split, parts, [&](int i, double u) {
                            return c <= i ? fma(wv[i], __ldcg(Kr + tri64(i) + c), u) : u;
                        });
                    part[tid] = v;
                    __syncthreads();
                    if (is == 0 && c <= nS) {
                        v = join_tree(part + ib * 32 + lane, nb * 32, split);
                        v = c == nS ? rd : -v * rd;
                        __stcg(Kr + tri64(nS) + c, v);
                        __stcg(Kc + column_at(c, k) + nS, v);
                        put_all<C>(xs + c, c == nS ? zn * v : fma(zn, v, xs[c]));
                    }
                    __syncthreads();
                }
            }
            if (tid == 0) {
                const uint32_t at = (haar ? (uint32_t)B : 0u) + jb % B;
                Sj[nS] = jb;
                prev[nS] = head[at];
                head[at] = (uint32_t)nS;
                fam_pos[haar ? k - 1 - nH : nC] = (uint32_t)nS;
                zs[nS] = zn;
            }
#pragma unroll
            for (int i = 0; i < 4 * EQ; ++i)
                if (is_here(i) && atom_of(i) == jb) taken |= 1u << i;
            if (haar) ++nH; else ++nC;
            ++nS;
            cluster_sync<C>();
        }

        // (a7) emit or split, as the MP kernel: CTA 0, which also tells the
        // others' near ties
        tie = __syncthreads_or(tie) != 0;
        if (tid == 0) {
            if (C == 1) offers[0].tie = tie ? 1.0 : 0.0;
            else put(&offers[rank].tie, 0u, tie ? 1.0 : 0.0);
        }
        cluster_sync<C>();
        bool tie_any = false;
        for (int r = 0; r < C; ++r) tie_any = tie_any || offers[r].tie != 0.0;
        const bool emit = conv || lv.is_last;
        if (rank == 0) {
            if (tid == 0) {
                atomicAdd(&a.ctr->attempts[lv.level], 1ull);
                atomicAdd(&a.ctr->iterations[lv.level], (unsigned long long)nS);
                atomicMax(&a.ctr->max_steps[lv.level], (unsigned)nS);
            }
            if (emit) {
                if (tid == 0) {
                    uint32_t off = kNoAtom, eslot = 0;
                    const unsigned long long slot = atomicAdd(&a.ctr->n_leaves, 1ull);
                    const unsigned long long o = atomicAdd(&a.ctr->n_atoms, (unsigned long long)nS);
                    const uint8_t flags = (uint8_t)((tie_any ? 1u : 0u) | (qe.flags & 2u));
                    if (slot >= a.leaf_cap || o + nS > a.atom_cap) {
                        raise_error(a.ctr, kDevErrQueueOverflow, 3u);
                    } else {
                        LeafRec rec;
                        rec.plane = qe.plane;
                        rec.y = qe.y;
                        rec.x = qe.x;
                        rec.atom_off = (uint32_t)o;
                        rec.b = (uint16_t)B;
                        rec.n_atoms = (uint16_t)nS;
                        rec.converged = conv ? 1 : 0;
                        rec.flags = flags;
                        rec.reserved = 0;
                        a.leaves[slot] = rec;
                        off = (uint32_t)o;
                        eslot = (uint32_t)slot;
                        const unsigned long long cell = cell_of(a.cells, a.planes[qe.plane], qe.y, qe.x);
                        if (cell != ~0ull) a.cells.cell[cell] = (uint32_t)slot + 1u;
                        if (flags) atomicAdd(&a.ctr->near_tie_leaves, 1ull);
                    }
                    bc[1] = off;
                    bc[2] = eslot;
                }
                __syncthreads();
                const uint32_t off = bc[1], eslot = bc[2];
                if (off != kNoAtom) {
                    for (int i = tid; i < nS; i += kThreads) {
                        const double x = xs[i];
                        const float hi = (float)x;
                        a.atoms[off + i] = AtomRec{Sj[i], hi};
                        a.alpha_lo[off + i] = (float)(x - (double)hi);
                        a.atom_leaf[off + i] = eslot;
                    }
                }
            } else if (tid == 0) {
                const unsigned slot = atomicAdd(lv.next_count, 4u);
                if (slot + 4u > lv.next_capacity) {
                    raise_error(a.ctr, kDevErrQueueOverflow, 4u);
                } else {
                    const uint32_t h = B / 2;
                    const uint32_t fl = (qe.flags & 2u) | (tie_any ? 2u : 0u);
                    lv.next_queue[slot + 0] = QueueEntry{qe.plane, qe.y, qe.x, fl};
                    lv.next_queue[slot + 1] = QueueEntry{qe.plane, qe.y, qe.x + h, fl};
                    lv.next_queue[slot + 2] = QueueEntry{qe.plane, qe.y + h, qe.x, fl};
                    lv.next_queue[slot + 3] = QueueEntry{qe.plane, qe.y + h, qe.x + h, fl};
                }
            }
        }
        cluster_sync<C>();
    }
}

unsigned long long omp_cta_slot_doubles(int k) { return k < 1 ? 0ull : (unsigned long long)slot_doubles(k); }

// A slot per cluster: as many as there are SMs or leaves.
unsigned long long omp_cta_workspace_doubles(int k, int sms, unsigned long long leaves) {
    const unsigned long long slots = leaves < (unsigned long long)sms ? leaves : (unsigned long long)sms;
    return slots * omp_cta_slot_doubles(k);
}

// C CTAs a leaf: the most that the level's leaves leave SMs for.
template <int B, int NF, int C>
static cudaError_t launch_omp_cta_c(const MPArgs &a, long long leaves, cudaStream_t st) {
    const int k = a.lv.k;
    const size_t bytes = OmpLayout<B, NF, C>::bytes(k);
    auto kern = omp_cta_kernel<B, NF, C>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.gridDim = dim3((unsigned)C, 1, 1);
    cfg.dynamicSmemBytes = bytes;
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = C > 1 ? 1 : 0;
    long long clusters = leaves;
    if (C > 1) {
        int most = 0;
        e = cudaOccupancyMaxActiveClusters(&most, kern, &cfg);
        if (e != cudaSuccess) return e;
        if constexpr (C > 1) {
            if (most < 1) return launch_omp_cta_c<B, NF, C / 2>(a, leaves, st);      // no room for a cluster this wide
        }
        if (most < clusters) clusters = most;
    }
    cfg.gridDim = dim3((unsigned)(clusters * C), 1, 1);
    return cudaLaunchKernelEx(&cfg, kern, a);
}

template <int B, int NF>
static cudaError_t launch_omp_cta_t(const MPArgs &a, cudaStream_t st) {
    const int k = a.lv.k;
    if (k < 1 || k > kMaxBudget || !a.omp_L || a.omp_sms < 1 || a.omp_L_doubles < omp_cta_slot_doubles(k))
        return cudaErrorInvalidValue;
    // the most leaves in flight: those there are, one an SM, one a slot
    const long long slots = (long long)(a.omp_L_doubles / omp_cta_slot_doubles(k));
    long long leaves = a.lv.capacity < 1u ? 1 : (long long)a.lv.capacity;
    if (leaves > a.omp_sms) leaves = a.omp_sms;
    if (leaves > slots) leaves = slots;
    if constexpr (NF == 2) {
        // A step's products shrink with C and its barriers and chains do not:
        // 16 leaves of side 64 took 7.69, 11.2, 18.7 and 33.3 ms with 8, 4, 2
        // CTAs and one, 64 leaves 8.0 with two against 14.5 with one.  More
        // CTAs than SMs would queue whole leaves
        if (B == 64 && leaves * 8 <= a.omp_sms) return launch_omp_cta_c<B, NF, (B == 64 ? 8 : 1)>(a, leaves, st);
        if (B == 64 && leaves * 4 <= a.omp_sms) return launch_omp_cta_c<B, NF, (B == 64 ? 4 : 1)>(a, leaves, st);
        if (leaves * 2 <= a.omp_sms) return launch_omp_cta_c<B, NF, 2>(a, leaves, st);
    }
    return launch_omp_cta_c<B, NF, 1>(a, leaves, st);
}

int omp_cta_max_budget() { return kMaxBudget; }


cudaError_t launch_omp_cta(const MPArgs &a, int nf, cudaStream_t st) {
    if (nf == 2) {
        switch (a.lv.b) {
            case 32: return launch_omp_cta_t<32, 2>(a, st);
            case 64: return launch_omp_cta_t<64, 2>(a, st);
        }
    } else {
        switch (a.lv.b) {
            case 32: return launch_omp_cta_t<32, 1>(a, st);
            case 64: return launch_omp_cta_t<64, 1>(a, st);
        }
    }
    return cudaErrorInvalidValue;
}

}  // namespace aqmp
