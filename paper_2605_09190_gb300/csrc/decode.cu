// decode.cu -- Algorithm 3 (mp_decoder): for every leaf of one plane,
// y = D_N x, un-ravel, and place the block at its position.  Each pixel
// sums alpha_t B[p_t][i] B[q_t][m] over the leaf's atoms in FP32 (the stored
// coefficients are FP32), in the order of the list; atoms listed twice simply
// add.
//
// The unit of work is a warp's tile of at most 256 pixels: 32 columns, one a
// lane, by 8 rows in a lane's registers.  Per atom a lane then loads its
// column's entry of row q once and the tile's 8 entries of row p as two
// broadcast 16-byte loads, for 8 products and 8 multiply-adds on the packed
// FP32 instructions -- where one thread per pixel took five loads for those
// two operations and was bound by the load pipe.  The 1-D bases of the sides
// up to 64 (43 KB) are copied to shared memory first: read through L1 their
// first touches are misses that each pursuit's random rows meet one by one.
// A side-64 leaf is sixteen tiles, a side-128 leaf 64, each on some other warp
// of the GPU, so that one leaf with many atoms does not outlast the rest.
// 1536x2048 RGB, 26 000 leaves a plane, three calls: 4.2 -> 0.43 ms.
#include <cuda_runtime.h>

#include "common.cuh"
#include "f32x2.cuh"
#include "kernels.h"
#include "leaf_tasks.cuh"

namespace aqmp {

namespace {

constexpr int kDecodeThreads = 256;
constexpr int kDecodeCtas = 3;                             // per SM
constexpr int kGroup = 4;                                  // atoms in flight

// Rows of a lane's tile column, and tiles of a leaf.
template <int B>
struct Tile {
    static constexpr int COLS = B < 32 ? B : 32;                   // columns across the lanes
    static constexpr int GROUPS = 32 / COLS;                       // row groups across the lanes (B < 32)
    static constexpr int ROWS = B >= 32 ? 8 : (B + GROUPS - 1) / GROUPS;    // rows in a lane's registers
    static constexpr int N = B >= 32 ? (B / 32) * (B / 8) : 1;     // tiles
};

constexpr int log2_of(int b) { return b <= 1 ? 0 : 1 + log2_of(b / 2); }

// Where side B's two bases start among those in shared memory (floats), and
// their total: sides 4, 8, 16, 32, 64.
constexpr int table_at(int b) { return b <= 4 ? 0 : table_at(b / 2) + 2 * (b / 2) * (b / 2); }
constexpr int kTableFloats = table_at(128);

// One tile of one leaf of side B.  stage: this warp's 32 atoms as (alpha,
// offset of row p, offset of row q) into the FP32 basis of their family;
// tables: the bases in shared memory (side 128: read through L1).
template <int B>
__device__ __forceinline__ void decode_tile(const DecodeArgs &a, const LeafRec &L, int tile, uint4 *stage,
                                            const float *tables) {
    using TL = Tile<B>;
    constexpr int n = B * B, R = TL::ROWS;
    const int lane = threadIdx.x & 31;
    const int m = B >= 32 ? tile % (B / 32) * 32 + lane : lane % TL::COLS;
    const int i0 = B >= 32 ? tile / (B / 32) * R : lane / TL::COLS * R;
    if (B < 32 && i0 >= B) return;                     // side 4 fills half a warp
    const unsigned peers = B == 4 ? 0x0000ffffu : 0xffffffffu;
    const int width = B == 4 ? 16 : 32;
    const float *basis = B <= 64 ? tables + table_at(B) : a.bases.basis[log2_of(B)];
    const float *colq = basis + m, *rowp = basis + i0;
    constexpr int P = R >= 2 ? R / 2 : 1;
    f2 acc[P];
#pragma unroll
    for (int r = 0; r < P; ++r) acc[r] = f2_make(0.0f, 0.0f);
    // the next batch of atoms is fetched while this one is applied
    AtomRec at{0u, 0.0f};
    auto fetch = [&](int t0) {
        if (t0 + lane < L.n_atoms) {
            at = a.atoms[L.atom_off + t0 + lane];
            if (a.alpha) at.alpha = a.alpha[L.atom_off + t0 + lane];
        }
    };
    if (lane < width) fetch(0);
    for (int t0 = 0; t0 < L.n_atoms; t0 += width) {
        const int cnt = min(width, (int)L.n_atoms - t0);
        int fam = (int)(at.j >= (uint32_t)n);
        const int f = (int)at.j - fam * n;
        if (a.bases.nf == 1) fam = a.bases.single_family;
        // past the last atom: nothing times entry 0
        stage[lane] = lane < cnt ? make_uint4(__float_as_uint(at.alpha), (uint32_t)(fam * n + (f % B) * B),
                                              (uint32_t)(fam * n + (f / B) * B), 0u)
                                 : make_uint4(0u, 0u, 0u, 0u);
        __syncwarp(peers);
        fetch(t0 + width);
        // all loads of a group of atoms before its arithmetic: a lone warp on a
        // long list is bound by their latency
#pragma unroll 1
        for (int t = 0; t < cnt; t += kGroup) {
            uint4 s[kGroup];
            float bq[kGroup];
            f2 bp[kGroup][P];
#pragma unroll
            for (int k = 0; k < kGroup; ++k) s[k] = stage[t + k];
#pragma unroll
            for (int k = 0; k < kGroup; ++k) {
                bq[k] = colq[s[k].z];
                const float *rp = rowp + s[k].y;
                if constexpr (R >= 4) {
#pragma unroll
                    for (int r = 0; r < R / 4; ++r) {
                        const ulonglong2 v = reinterpret_cast<const ulonglong2 *>(rp)[r];
                        bp[k][2 * r] = v.x;
                        bp[k][2 * r + 1] = v.y;
                    }
                } else if constexpr (R == 2) {
                    bp[k][0] = *reinterpret_cast<const f2 *>(rp);
                } else {
                    bp[k][0] = f2_make(rp[0], 0.0f);
                }
            }
#pragma unroll
            for (int k = 0; k < kGroup; ++k) {
                const float al = __uint_as_float(s[k].x);
                const f2 al2 = f2_make(al, al), bq2 = f2_make(bq[k], bq[k]);
#pragma unroll
                for (int r = 0; r < P; ++r) acc[r] = f2_fma(al2, f2_mul(bp[k][r], bq2), acc[r]);
            }
        }
        __syncwarp(peers);
    }
    const int i = (int)(L.plane - a.out.plane);
    const long long pitch = a.out.pitch[i];
    float *out = a.out.img[i] + (long long)(L.y + i0) * pitch + L.x + m;
#pragma unroll
    for (int r = 0; r < R; ++r) out[r * pitch] = r & 1 ? f2_y(acc[r / 2]) : f2_x(acc[r / 2]);
}

}  // namespace

// All tiles of a leaf on one CTA: the busiest SM worked 1.7 times as long as
// the mean; scattered over the GPU (leaf_tasks.cuh) they balance.
__global__ void __launch_bounds__(kDecodeThreads, kDecodeCtas) decode_kernel(const __grid_constant__ DecodeArgs a, unsigned tiles) {
    extern __shared__ __align__(16) unsigned char smem[];
    float *tables = reinterpret_cast<float *>(smem);
    uint4 *stage = reinterpret_cast<uint4 *>(tables + kTableFloats) + (threadIdx.x & ~31u);
    __shared__ unsigned long long s_range[2];
    const int warp = threadIdx.x >> 5;
    // the bases of the code's sides (one or two families)
#pragma unroll 1
    for (int lg = 2, at = 0; lg <= 6; ++lg) {
        const int bb = 1 << (2 * lg);
        if (a.bases.basis[lg] != nullptr)
            for (int i = threadIdx.x; i < bb / 2; i += kDecodeThreads)
                reinterpret_cast<float4 *>(tables + at)[i] = reinterpret_cast<const float4 *>(a.bases.basis[lg])[i];
        at += 2 * bb;
    }
    if (warp < 2) {
        const uint32_t plane = a.out.plane + (uint32_t)(warp ? a.out.n_planes : 0);
        const unsigned long long at = first_of_plane(a.leaves, a.n_leaves, plane);
        if ((threadIdx.x & 31) == 0) s_range[warp] = at;
    }
    __syncthreads();
    for_tiles(
        a.leaves, s_range[0], (unsigned)(s_range[1] - s_range[0]), tiles, blockIdx.x + gridDim.x * (unsigned)warp,
        gridDim.x * (kDecodeThreads / 32), [](int b) { return b >= 32 ? (b / 32) * (b / 8) : 1; },
        [&](const LeafRec &L, unsigned long long, int tile) {
            switch (L.b) {
                case 4: decode_tile<4>(a, L, tile, stage, tables); break;
                case 8: decode_tile<8>(a, L, tile, stage, tables); break;
                case 16: decode_tile<16>(a, L, tile, stage, tables); break;
                case 32: decode_tile<32>(a, L, tile, stage, tables); break;
                case 64: decode_tile<64>(a, L, tile, stage, tables); break;
                case 128: decode_tile<128>(a, L, tile, stage, tables); break;
                default: break;
            }
            __syncwarp();
        });
}

cudaError_t launch_decode(const DecodeArgs &a, int num_sms, cudaStream_t st) {
    if (a.n_leaves == 0) return cudaSuccess;
    const float *const *basis = a.bases.basis;
    const unsigned tiles = basis[7] ? Tile<128>::N : basis[6] ? Tile<64>::N : basis[5] ? Tile<32>::N : 1u;
    unsigned long long blocks = (a.n_leaves * tiles + kDecodeThreads / 32 - 1) / (kDecodeThreads / 32);
    const unsigned long long cap = (unsigned long long)num_sms * kDecodeCtas;
    if (blocks > cap) blocks = cap;
    constexpr size_t smem = sizeof(float) * kTableFloats + sizeof(uint4) * kDecodeThreads;
    cudaError_t e = cudaFuncSetAttribute(decode_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    decode_kernel<<<(unsigned)blocks, kDecodeThreads, smem, st>>>(a, tiles);
    return cudaGetLastError();
}

}  // namespace aqmp
