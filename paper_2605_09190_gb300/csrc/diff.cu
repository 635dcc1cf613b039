// diff.cu -- the adjoint of the sparse synthesis (Algorithm 3 with caller
// coefficients on a fixed MP support), for the refinement.
//
// Synthesis: recon[y+i][x+m] = sum_t alpha_t B[p_t][i] B[q_t][m] per leaf
// (decode.cu).  Adjoint: d recon / d alpha_t is the atom itself, so
// grad alpha_t = <G_leaf, phi_t> for the leaf's block G of the incoming
// gradient = (B G B^T)[p_t][q_t]: U = B G, T = U B^T per family, then a gather
// at the leaf's atoms.  FP32, each entry summed in ascending order.
//
// Sides up to 32 take a warp per leaf, 64 and 128 a CTA.  A lane computes
// tiles of 4 x 4 entries (2 x 2 at side 8, one at side 4), so 64 multiply-adds
// share eight 16-byte loads -- one entry at a time took two loads for each
// multiply-add and was bound by the load pipe.  Stage 1's lanes run along m
// (rows of B broadcast, rows of G contiguous), stage 2's along p (rows of B
// broadcast again, rows of U in a layout that spreads their 16-byte words over
// the banks), so no transposed copy of the basis is needed.
// 16 planes of 512x512, sides 32..8: 2.2 ms in 16 launches -> 75 us in one.
#include <cuda_runtime.h>

#include "common.cuh"
#include "kernels.h"
#include "leaf_tasks.cuh"

namespace aqmp {

namespace {

constexpr int kWarpThreads = 256;                         // of the warp-per-leaf kernel
constexpr int kWarpFloats = 3 * 32 * 32;                  // G, U, T of side 32; sides <= 16: G, two each
constexpr int kCtaThreads = 256;

template <int B>
constexpr int tile_edge() { return B >= 16 ? 4 : B == 8 ? 2 : 1; }

// Word of U[p][m]: 16-byte words of a row exchanged by its tile row, so that
// the tiles of a column of tiles lie in different banks.
template <int B>
__device__ __forceinline__ int u_at(int p, int m) {
    return B >= 16 ? p * B + ((((m >> 2) ^ (p >> 2)) & (B / 4 - 1)) << 2) + (m & 3) : p * B + m;
}

template <int N>
__device__ __forceinline__ void load_n(const float *src, float (&v)[N]) {
    if constexpr (N == 4) {
        const float4 x = *reinterpret_cast<const float4 *>(src);
        v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
    } else if constexpr (N == 2) {
        const float2 x = *reinterpret_cast<const float2 *>(src);
        v[0] = x.x; v[1] = x.y;
    } else {
        v[0] = *src;
    }
}

template <int N>
__device__ __forceinline__ void store_n(float *dst, const float (&v)[N]) {
    if constexpr (N == 4) *reinterpret_cast<float4 *>(dst) = make_float4(v[0], v[1], v[2], v[3]);
    else if constexpr (N == 2) *reinterpret_cast<float2 *>(dst) = make_float2(v[0], v[1]);
    else *dst = v[0];
}

// U = Bf G, thread `t` of NT.
template <int B, int NT>
__device__ __forceinline__ void stage1(const float *Bf, const float *G, float *U, int t) {
    constexpr int E = tile_edge<B>(), TB = B / E;
    for (int tile = t; tile < TB * TB; tile += NT) {
        const int p0 = tile / TB * E, m0 = tile % TB * E;
        float s[E][E];
#pragma unroll
        for (int r = 0; r < E; ++r)
#pragma unroll
            for (int c = 0; c < E; ++c) s[r][c] = 0.0f;
#pragma unroll 4
        for (int i = 0; i < B; i += 4) {
            float b[E][4], g[4][E];
#pragma unroll
            for (int r = 0; r < E; ++r) load_n<4>(Bf + (p0 + r) * B + i, b[r]);
#pragma unroll
            for (int k = 0; k < 4; ++k) load_n<E>(G + (i + k) * B + m0, g[k]);
#pragma unroll
            for (int k = 0; k < 4; ++k)
#pragma unroll
                for (int r = 0; r < E; ++r)
#pragma unroll
                    for (int c = 0; c < E; ++c) s[r][c] = __fmaf_rn(b[r][k], g[k][c], s[r][c]);
        }
#pragma unroll
        for (int r = 0; r < E; ++r) store_n<E>(U + u_at<B>(p0 + r, m0), s[r]);
    }
}

// T[q][p] = (U Bf^T)[p][q].
template <int B, int NT>
__device__ __forceinline__ void stage2(const float *Bf, const float *U, float *T, int t) {
    constexpr int E = tile_edge<B>(), TB = B / E;
    for (int tile = t; tile < TB * TB; tile += NT) {
        const int p0 = tile % TB * E, q0 = tile / TB * E;
        float s[E][E];                                     // [q][p]
#pragma unroll
        for (int r = 0; r < E; ++r)
#pragma unroll
            for (int c = 0; c < E; ++c) s[c][r] = 0.0f;
#pragma unroll 4
        for (int m = 0; m < B; m += 4) {
            float u[E][4], b[E][4];
#pragma unroll
            for (int r = 0; r < E; ++r) load_n<4>(U + u_at<B>(p0 + r, m), u[r]);
#pragma unroll
            for (int c = 0; c < E; ++c) load_n<4>(Bf + (q0 + c) * B + m, b[c]);
#pragma unroll
            for (int k = 0; k < 4; ++k)
#pragma unroll
                for (int r = 0; r < E; ++r)
#pragma unroll
                    for (int c = 0; c < E; ++c) s[c][r] = __fmaf_rn(u[r][k], b[c][k], s[c][r]);
        }
#pragma unroll
        for (int c = 0; c < E; ++c) store_n<E>(T + (q0 + c) * B + p0, s[c]);
    }
}

template <int NT>
__device__ __forceinline__ void sync_group() {
    if (NT <= 32) __syncwarp();
    else __syncthreads();
}

// One leaf on NT threads; sm: 3 b^2 floats (5 b^2 up to side 16, where the two
// families run side by side on half of the warp each).
template <int B, int NT>
__device__ __forceinline__ void adjoint_leaf(const AdjointArgs &a, const LeafRec &L, float *sm, int t) {
    constexpr int n = B * B, LG = B == 4 ? 2 : B == 8 ? 3 : B == 16 ? 4 : B == 32 ? 5 : B == 64 ? 6 : 7;
    constexpr bool BOTH = B <= 16;
    if (L.n_atoms == 0) return;
    const int nfam = a.bases.nf, img = (int)(L.plane - a.grad.plane);
    const long long pitch = a.grad.pitch[img];
    const float *src = a.grad.img[img] + (long long)L.y * pitch + L.x;
    float *G = sm, *U = G + n, *T = U + (BOTH ? 2 * n : n);
#pragma unroll 8
    for (int v = t; v < n; v += NT) G[v] = src[(long long)(v / B) * pitch + v % B];
    sync_group<NT>();
    const float *basis = a.bases.basis[LG] + (nfam == 1 ? a.bases.single_family * n : 0);
    const AtomRec *atoms = a.atoms + L.atom_off;
    float *out = a.grad_alpha + L.atom_off;
    if constexpr (BOTH) {
        const int fam = t / (NT / 2), ft = t % (NT / 2);
        if (fam < nfam) stage1<B, NT / 2>(basis + fam * n, G, U + fam * n, ft);
        sync_group<NT>();
        if (fam < nfam) stage2<B, NT / 2>(basis + fam * n, U + fam * n, T + fam * n, ft);
        sync_group<NT>();
        for (int i = t; i < L.n_atoms; i += NT) {
            const uint32_t j = atoms[i].j;
            if (j < (uint32_t)(nfam * n)) out[i] = T[j];       // T[fam][q][p] at fam n + q b + p
        }
    } else {
        for (int fam = 0; fam < nfam; ++fam) {
            stage1<B, NT>(basis + fam * n, G, U, t);
            sync_group<NT>();
            stage2<B, NT>(basis + fam * n, U, T, t);
            sync_group<NT>();
            for (int i = t; i < L.n_atoms; i += NT) {
                const uint32_t f = atoms[i].j - (uint32_t)(fam * n);
                if (f < (uint32_t)n) out[i] = T[f];
            }
        }
    }
    sync_group<NT>();
}

__device__ __forceinline__ void plane_range(const AdjointArgs &a, unsigned long long (&range)[2]) {
    const int warp = threadIdx.x >> 5;
    if (warp < 2) {
        const uint32_t plane = a.grad.plane + (uint32_t)(warp ? a.grad.n_planes : 0);
        const unsigned long long at = first_of_plane(a.leaves, a.n_leaves, plane);
        if ((threadIdx.x & 31) == 0) range[warp] = at;
    }
    __syncthreads();
}

// Leaves of side <= 32, a warp each.
__global__ void __launch_bounds__(kWarpThreads) adjoint_warp_kernel(const __grid_constant__ AdjointArgs a) {
    extern __shared__ __align__(16) float sm_all[];
    __shared__ unsigned long long range[2];
    plane_range(a, range);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float *sm = sm_all + warp * kWarpFloats;
    for_tiles(
        a.leaves, range[0], (unsigned)(range[1] - range[0]), 1u, blockIdx.x + gridDim.x * (unsigned)warp,
        gridDim.x * (kWarpThreads / 32), [](int b) { return b <= 32 ? 1 : 0; },
        [&](const LeafRec &L, unsigned long long, int) {
            switch (L.b) {
                case 4: adjoint_leaf<4, 32>(a, L, sm, lane); break;
                case 8: adjoint_leaf<8, 32>(a, L, sm, lane); break;
                case 16: adjoint_leaf<16, 32>(a, L, sm, lane); break;
                case 32: adjoint_leaf<32, 32>(a, L, sm, lane); break;
                default: break;
            }
        });
}

// Leaves of side 64 and 128, a CTA each: leaves blockIdx.x + gridDim.x i, 256
// of them looked over at a time.
__global__ void __launch_bounds__(kCtaThreads) adjoint_cta_kernel(const __grid_constant__ AdjointArgs a) {
    extern __shared__ __align__(16) float sm_all[];
    __shared__ unsigned long long range[2];
    __shared__ unsigned list[kCtaThreads], found;
    plane_range(a, range);
    const unsigned count = (unsigned)(range[1] - range[0]);
    for (unsigned long long base = blockIdx.x; base < count; base += (unsigned long long)gridDim.x * kCtaThreads) {
        if (threadIdx.x == 0) found = 0u;
        __syncthreads();
        const unsigned long long at = base + (unsigned long long)gridDim.x * threadIdx.x;
        if (at < count && a.leaves[range[0] + at].b >= 64) list[atomicAdd(&found, 1u)] = (unsigned)at;
        __syncthreads();
        for (unsigned i = 0; i < found; ++i) {
            const LeafRec L = a.leaves[range[0] + list[i]];
            if (L.b == 64) adjoint_leaf<64, kCtaThreads>(a, L, sm_all, (int)threadIdx.x);
            else if (L.b == 128) adjoint_leaf<128, kCtaThreads>(a, L, sm_all, (int)threadIdx.x);
        }
        __syncthreads();
    }
}

}  // namespace

cudaError_t launch_synth_backward(const AdjointArgs &a, int num_sms, cudaStream_t st) {
    if (a.n_leaves == 0) return cudaSuccess;
    cudaError_t e = cudaSuccess;
    const float *const *basis = a.bases.basis;
    if (basis[2] || basis[3] || basis[4] || basis[5]) {
        constexpr size_t smem = sizeof(float) * kWarpFloats * (kWarpThreads / 32);
        e = cudaFuncSetAttribute(adjoint_warp_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        unsigned long long blocks = (a.n_leaves + kWarpThreads / 32 - 1) / (kWarpThreads / 32);
        if (blocks > (unsigned long long)num_sms * 2) blocks = (unsigned long long)num_sms * 2;
        adjoint_warp_kernel<<<(unsigned)blocks, kWarpThreads, smem, st>>>(a);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    if (basis[6] || basis[7]) {
        const size_t side = basis[7] ? 128 : 64, smem = sizeof(float) * 3 * side * side;
        e = cudaFuncSetAttribute(adjoint_cta_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        unsigned long long blocks = a.n_leaves;
        const unsigned long long cap = (unsigned long long)num_sms * (basis[7] ? 1 : 4);
        if (blocks > cap) blocks = cap;
        adjoint_cta_kernel<<<(unsigned)blocks, kCtaThreads, smem, st>>>(a);
        e = cudaGetLastError();
    }
    return e;
}

}  // namespace aqmp
