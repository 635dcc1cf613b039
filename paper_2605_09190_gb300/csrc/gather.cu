// gather.cu -- (a1) block gather and the level-0 root queue.
//
// A leaf vector is the column-major unravel of its block (Appendix A:
// concatenate the columns): element v = m b + i holds pixel (row i, col m).
// The correlation kernels take it centred, y - 128, as BF16: every value in
// [-128, 127] is exact in BF16; the centring is undone exactly inside the
// correlation by adding 128 sum_v D_fix[j][v].  The BF16 form with rescore
// centres on the block's mean rounded to an integer instead (values in
// [-255, 255], still exact in BF16), recorded per leaf.
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <cuda_fp8.h>

#include "common.cuh"
#include "kernels.h"

namespace aqmp {

// The gather of a leaf as BF16 and its sum of squares, for a queue's entries
// or (queue NULL) for contiguous row-major blocks.  A thread takes 4 x 4
// pixels: four words of four rows in, and, pairing the rows' bytes of one
// column, four stores of four consecutive elements v out.  A warp covers 16
// rows x 32 columns, so loads and stores both fill 32-byte sectors and nothing
// goes through shared memory.  (B / 4)^2 / 32 warps a leaf, 8 at the most; at
// sides 4 to 16 a warp takes several leaves.  HBM bounds it.  50 910 leaves of
// side 64 (626 MB) take 0.128 ms, 4.9 TB/s, and 0.393 before (bytes through a
// transposed tile); 3072 of side 128 0.033 ms and 0.107.
// Planes whose address or pitch is no multiple of 4 are read by bytes.
struct GatherSource {
    const QueueEntry *queue;
    const PlaneDesc *planes;
    const unsigned *count;
    const uint8_t *blocks;
    long long n_blocks;
};

template <int B>
__global__ void __launch_bounds__(256)
gather_kernel(GatherSource s, int Kpad, __nv_bfloat16 *__restrict__ Y, uint32_t *e0, uint8_t *mu) {
    constexpr int n = B * B, IB = B / 4, U = IB * IB;             // 4 x 4 units of a leaf
    constexpr int TPL = U < 256 ? (U > 32 ? 32 : U) : 256;        // threads a leaf
    constexpr int UPT = U / TPL, GROUPS = 256 / TPL;
    constexpr int LI = IB < 4 ? IB : 4, LM = (TPL < 32 ? TPL : 32) / LI;   // a warp's units along i and m
    __shared__ uint32_t s_sum[2][2][8];
    const int t = threadIdx.x % TPL;
    const long long count = s.queue ? (long long)*s.count : s.n_blocks;
    const long long step = (long long)gridDim.x * GROUPS;
    int turn = 0;
    // a group's leaf may be past the end: its lanes stay for the shuffles
    for (long long first = (long long)blockIdx.x * GROUPS; first < count; first += step, turn ^= 1) {
        const long long leaf = first + threadIdx.x / TPL;
        const bool live = leaf < count;
        uint32_t w[UPT][4] = {}, ss = 0, sy = 0;
        int ib[UPT], mb[UPT];
#pragma unroll
        for (int k = 0; k < UPT; ++k) {
            const int u = t + k * TPL, tile = u / (LI * LM), l = u % (LI * LM);
            ib[k] = (tile % (IB / LI)) * LI + l % LI;
            mb[k] = (tile / (IB / LI)) * LM + l / LI;
        }
        if (live) {
            const uint8_t *base;
            long long pitch;
            if (s.queue) {
                const QueueEntry q = s.queue[leaf];
                const PlaneDesc pd = s.planes[q.plane];
                pitch = pd.pitch;
                base = pd.pix + (long long)q.y * pitch + q.x;
            } else {
                pitch = B;
                base = s.blocks + leaf * n;
            }
            if ((((unsigned long long)base | (unsigned long long)pitch) & 3ull) == 0ull) {
#pragma unroll
                for (int k = 0; k < UPT; ++k)
#pragma unroll
                    for (int r = 0; r < 4; ++r)
                        w[k][r] = *reinterpret_cast<const uint32_t *>(base + (4 * ib[k] + r) * pitch + 4 * mb[k]);
            } else {
#pragma unroll 1
                for (int k = 0; k < UPT; ++k)
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        const uint8_t *p = base + (4 * ib[k] + r) * pitch + 4 * mb[k];
                        const uint32_t x = p[0] | (uint32_t)p[1] << 8 | (uint32_t)p[2] << 16 | (uint32_t)p[3] << 24;
#pragma unroll
                        for (int i = 0; i < UPT; ++i)
                            if (i == k) w[i][r] = x;
                    }
            }
#pragma unroll
            for (int k = 0; k < UPT; ++k)
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    ss = __dp4a(w[k][r], w[k][r], ss);
                    sy = __dp4a(w[k][r], 0x01010101u, sy);
                }
        }
#pragma unroll
        for (int off = (TPL < 32 ? TPL : 32) / 2; off > 0; off >>= 1) {
            ss += __shfl_xor_sync(0xffffffffu, ss, off);
            sy += __shfl_xor_sync(0xffffffffu, sy, off);
        }
        if (TPL == 256) {
            if ((threadIdx.x & 31) == 0) {
                s_sum[turn][0][threadIdx.x >> 5] = ss;
                s_sum[turn][1][threadIdx.x >> 5] = sy;
            }
            __syncthreads();                                     // the other turn's readers are past this one
            ss = sy = 0;
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                ss += s_sum[turn][0][i];
                sy += s_sum[turn][1][i];
            }
        }
        if (!live) continue;
        // the centre: 128, or (BF16 form with rescore) the block's mean
        // rounded to an integer, so that y - centre stays exact in BF16
        uint32_t shift = 0;
        if (mu) {
            const int centre = (int)((sy + (uint32_t)(n / 2)) / (uint32_t)n);
            if (t == 0) mu[leaf] = (uint8_t)centre;
            const __nv_bfloat16 d = __float2bfloat16_rn((float)(128 - centre));
            shift = (uint32_t)__bfloat16_as_ushort(d) * 0x10001u;
        }
        if (t == 0 && e0) e0[leaf] = ss;
        __nv_bfloat16 *dst = Y + leaf * Kpad;
#pragma unroll
        for (int k = 0; k < UPT; ++k)
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                uint2 v = make_uint2(bytes_less_128(w[k][0], w[k][1], c), bytes_less_128(w[k][2], w[k][3], c));
                if (mu) {
                    asm("add.rn.bf16x2 %0, %0, %1;" : "+r"(v.x) : "r"(shift));
                    asm("add.rn.bf16x2 %0, %0, %1;" : "+r"(v.y) : "r"(shift));
                }
                *reinterpret_cast<uint2 *>(dst + (4 * mb[k] + c) * B + 4 * ib[k]) = v;
            }
        for (int v = n + 4 * t; v < Kpad; v += 4 * TPL) *reinterpret_cast<uint2 *>(dst + v) = make_uint2(0u, 0u);
    }
}

template <int B>
static cudaError_t launch_gather_t(const GatherSource &s, long long capacity, int Kpad, __nv_bfloat16 *Y, uint32_t *e0,
                                   uint8_t *mu, int num_sms, cudaStream_t st) {
    constexpr int U = (B / 4) * (B / 4), GROUPS = U >= 256 ? 1 : 256 / (U > 32 ? 32 : U);
    long long blocks = (capacity + GROUPS - 1) / GROUPS;
    const long long cap = (long long)num_sms * 8;
    if (blocks > cap) blocks = cap;
    if (blocks < 1) blocks = 1;
    gather_kernel<B><<<(unsigned)blocks, 256, 0, st>>>(s, Kpad, Y, e0, mu);
    return cudaGetLastError();
}

static cudaError_t launch_gather_bf16(int b, const GatherSource &s, long long capacity, int Kpad, __nv_bfloat16 *Y,
                                      uint32_t *e0, uint8_t *mu, int num_sms, cudaStream_t st) {
    switch (b) {
        case 4: return launch_gather_t<4>(s, capacity, Kpad, Y, e0, mu, num_sms, st);
        case 8: return launch_gather_t<8>(s, capacity, Kpad, Y, e0, mu, num_sms, st);
        case 16: return launch_gather_t<16>(s, capacity, Kpad, Y, e0, mu, num_sms, st);
        case 32: return launch_gather_t<32>(s, capacity, Kpad, Y, e0, mu, num_sms, st);
        case 64: return launch_gather_t<64>(s, capacity, Kpad, Y, e0, mu, num_sms, st);
        case 128: return launch_gather_t<128>(s, capacity, Kpad, Y, e0, mu, num_sms, st);
    }
    return cudaErrorInvalidValue;
}

// The FP8 form's gather: TPL threads per leaf (a warp below side 32, the whole 256-thread CTA at
// sides 32 to 128), grid-stride over the level's entries.  The block's rows
// are read coalesced into the group's shared-memory tile (row stride B + 4
// bytes), then written in unravel order v = m B + i as E4M3 bytes, so both
// the pixel reads and the writes are contiguous.
template <int B, int TPL>
__global__ void __launch_bounds__(256) gather_fp8_kernel(GatherArgs a) {
    constexpr int n = B * B, stride = B + 4, GROUPS = 256 / TPL, NW = TPL / 32;
    extern __shared__ uint8_t gather_tile[];
    __shared__ uint32_t s_ss[8];
    const int t = threadIdx.x % TPL, g = threadIdx.x / TPL, lane = threadIdx.x & 31;
    uint8_t *tile = gather_tile + (size_t)g * B * stride;
    const unsigned count = *a.count;
    for (unsigned leaf = blockIdx.x * GROUPS + g; leaf < count; leaf += gridDim.x * GROUPS) {
        const QueueEntry q = a.queue[leaf];
        const PlaneDesc pd = a.planes[q.plane];
        const uint8_t *base = pd.pix + (long long)q.y * pd.pitch + q.x;
        uint32_t ss = 0;
#pragma unroll 4
        for (int idx = t; idx < n; idx += TPL) {               // rows, coalesced
            const int i = idx / B, m = idx % B;
            const uint32_t p = base[(long long)i * pd.pitch + m];
            ss += p * p;
            tile[i * stride + m] = (uint8_t)p;
        }
        if (TPL == 32) __syncwarp(); else __syncthreads();
        {
            // FP8 form: centred pixels times the block's power-of-two scale
            // s_l (the largest with max |y~| s_l <= 448), rounded to E4M3
            uint32_t amax = 0;
            for (int idx = t; idx < n; idx += TPL) {
                const int d = (int)tile[(idx / B) * stride + idx % B] - 128;
                amax = max(amax, (uint32_t)(d < 0 ? -d : d));
            }
            for (int off = 16; off > 0; off >>= 1) amax = max(amax, __shfl_xor_sync(0xffffffffu, amax, off));
            if (NW > 1) {
                if (lane == 0) s_ss[threadIdx.x >> 5] = amax;
                __syncthreads();
                amax = 0;
                for (int w = 0; w < NW; ++w) amax = max(amax, s_ss[w]);
                __syncthreads();
            }
            int ex = 0;
            while (amax > 0 && ((unsigned long long)amax << (ex + 1)) <= 448ull) ++ex;
            const float sl = (float)(1 << ex);
            const int K8 = kpad_fp8(n);
            uint8_t *dst8 = a.Y8 + (size_t)leaf * K8;
            for (int v = t; v < K8; v += TPL) {
                __nv_fp8_storage_t q8 = 0;
                if (v < n)
                    q8 = __nv_cvt_float_to_fp8((float)((int)tile[(v % B) * stride + v / B] - 128) * sl,
                                               __NV_SATFINITE, __NV_E4M3);
                dst8[v] = q8;
            }
            if (t == 0) a.inv_sl[leaf] = 1.0f / sl;
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, off);
        if (NW == 1) {
            if (lane == 0) a.e0[leaf] = ss;
            __syncwarp();
        } else {
            if (lane == 0) s_ss[threadIdx.x >> 5] = ss;
            __syncthreads();
            if (threadIdx.x == 0) {
                uint32_t tot = 0;
                for (int w = 0; w < NW; ++w) tot += s_ss[w];
                a.e0[leaf] = tot;
            }
            __syncthreads();
        }
    }
}

template <int B>
static cudaError_t launch_gather_fp8_t(const GatherArgs &a, int num_sms, cudaStream_t st) {
    constexpr int TPL = B >= 32 ? 256 : 32;
    constexpr int GROUPS = 256 / TPL;
    long long blocks = ((long long)a.capacity + GROUPS - 1) / GROUPS;
    const long long cap = (long long)num_sms * 8;
    if (blocks > cap) blocks = cap;
    if (blocks < 1) blocks = 1;
    const size_t smem = (size_t)GROUPS * B * (B + 4);
    gather_fp8_kernel<B, TPL><<<(unsigned)blocks, 256, smem, st>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_gather(const GatherArgs &a, int num_sms, cudaStream_t st) {
    if (!a.Y8)
        return launch_gather_bf16(a.b, GatherSource{a.queue, a.planes, a.count, nullptr, 0}, a.capacity, a.Kpad, a.Y, a.e0,
                                  a.mu, num_sms, st);
    switch (a.b) {
        case 4: return launch_gather_fp8_t<4>(a, num_sms, st);
        case 8: return launch_gather_fp8_t<8>(a, num_sms, st);
        case 16: return launch_gather_fp8_t<16>(a, num_sms, st);
        case 32: return launch_gather_fp8_t<32>(a, num_sms, st);
        case 64: return launch_gather_fp8_t<64>(a, num_sms, st);
        case 128: return launch_gather_fp8_t<128>(a, num_sms, st);
    }
    return cudaErrorInvalidValue;
}

// L contiguous row-major b x b blocks (centred on 128, or with `mu` on each
// block's integer mean, recorded in mu[leaf]).
cudaError_t launch_gather_blocks(int b, int Kpad, const uint8_t *blocks, long long L,
                                 __nv_bfloat16 *Y, uint32_t *e0, int num_sms, cudaStream_t st, uint8_t *mu) {
    return launch_gather_bf16(b, GatherSource{nullptr, nullptr, nullptr, blocks, L}, L, Kpad, Y, e0, mu, num_sms, st);
}

// The same for the FP8 form: e4m3(y~ s_l) with the block's power-of-two
// scale s_l (max |y~| s_l <= 448), zero padded to kpad_fp8(n), and 1 / s_l.
__global__ void gather_blocks_fp8_kernel(int b, const uint8_t *blocks, long long L, uint8_t *Y8, float *inv_sl) {
    const int lane = threadIdx.x & 31;
    const long long warps = ((long long)gridDim.x * blockDim.x) >> 5;
    const int n = b * b, K8 = kpad_fp8(n);
    for (long long leaf = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; leaf < L; leaf += warps) {
        const uint8_t *base = blocks + leaf * n;
        uint32_t amax = 0;
        for (int v = lane; v < n; v += 32) {
            const int d = (int)base[v] - 128;
            amax = max(amax, (uint32_t)(d < 0 ? -d : d));
        }
        for (int off = 16; off > 0; off >>= 1) amax = max(amax, __shfl_xor_sync(0xffffffffu, amax, off));
        int ex = 0;
        while (amax > 0 && ((unsigned long long)amax << (ex + 1)) <= 448ull) ++ex;
        const float sl = (float)(1 << ex);
        for (int v = lane; v < K8; v += 32) {
            __nv_fp8_storage_t q8 = 0;
            if (v < n) {
                const int m = v / b, i = v - m * b;
                q8 = __nv_cvt_float_to_fp8((float)((int)base[i * b + m] - 128) * sl, __NV_SATFINITE, __NV_E4M3);
            }
            Y8[leaf * K8 + v] = q8;
        }
        if (lane == 0) inv_sl[leaf] = 1.0f / sl;
    }
}

cudaError_t launch_gather_blocks_fp8(int b, const uint8_t *blocks, long long L, uint8_t *Y8, float *inv_sl,
                                     int num_sms, cudaStream_t st) {
    long long blocks_needed = (L + 7) / 8;
    long long cap = (long long)num_sms * 8;
    if (blocks_needed > cap) blocks_needed = cap;
    if (blocks_needed < 1) blocks_needed = 1;
    gather_blocks_fp8_kernel<<<(unsigned)blocks_needed, 256, 0, st>>>(b, blocks, L, Y8, inv_sl);
    return cudaGetLastError();
}

// Roots of every plane in row-major order (Algorithm 1 loops over channels;
// Algorithm 2 starts from the N_max blocks of each).
__global__ void seed_roots_kernel(const PlaneDesc *planes, int n_planes, int max_block,
                                  unsigned total, QueueEntry *queue, unsigned *count) {
    for (unsigned r = blockIdx.x * blockDim.x + threadIdx.x; r < total; r += gridDim.x * blockDim.x) {
        int p = 0;
        while (p + 1 < n_planes && planes[p + 1].root_off <= r) ++p;
        const unsigned local = r - planes[p].root_off;
        const unsigned ry = local / planes[p].roots_x, rx = local - ry * planes[p].roots_x;
        queue[r] = QueueEntry{(uint32_t)p, ry * (uint32_t)max_block, rx * (uint32_t)max_block, 0u};
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) *count = total;
}

cudaError_t launch_seed_roots(const PlaneDesc *planes, int n_planes, int max_block,
                              unsigned total_roots, QueueEntry *queue, unsigned *count,
                              cudaStream_t st) {
    unsigned blocks = (total_roots + 255) / 256;
    if (blocks < 1) blocks = 1;
    if (blocks > 4096) blocks = 4096;
    seed_roots_kernel<<<blocks, 256, 0, st>>>(planes, n_planes, max_block, total_roots, queue, count);
    return cudaGetLastError();
}

}  // namespace aqmp
