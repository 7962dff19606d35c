// FP32 search of the projection P = D X^T (Sec. IV-A) with the selection
// i* = argmax_i |<g_i, r>| (Sec. III-A) fused: an HBM-bound GEMV over the
// stored FP32 dictionary.
#include <cuda_runtime.h>
#include <stdint.h>

#include "act_device.cuh"
#include "act_internal.cuh"

namespace act {

// ---------------------------------------------------------------------------
// FP32 GEMV over the stored dictionary with the selection fused.
// ---------------------------------------------------------------------------
// Each warp owns rows gw, gw + nw, gw + 2 nw, ... (nw = warps in the grid)
// and streams two rows at a time with 128-bit loads: lane l reads float4
// l + 32 j of a row, j = 0..NV-1.  The residual is brought into shared memory
// by the TMA bulk-copy engine and then held in registers; several channels
// (the queue of a tensor-core search's full searches) follow one another.  A
// warp-shuffle reduction gives every lane the row's score; the warp keeps its
// best |score| (lowest row on ties, rows are visited in increasing order),
// the block combines its warps and issues one 64-bit atomicMax of the packed
// key per channel.  With WRITE every score is stored instead (the projection
// of one channel, project_multi_bytes, or of few, one_by_one).
template <int NV, bool WRITE>
__global__ void __launch_bounds__(kGemvThreads) k_gemv(const float *__restrict__ D, int64_t K, int Lp,
                                                       const float *R, int B, const int *chlist, const int *count_dev,
                                                       unsigned long long *keys, float *scores, int *status,
                                                       unsigned long long wait_ns) {
    extern __shared__ __align__(128) float smem_r[];  // Lp floats
    __shared__ __align__(8) uint64_t bar;
    __shared__ float red_s[kGemvThreads / 32];
    __shared__ uint32_t red_i[kGemvThreads / 32];

    // launched as a programmatic dependent of the kernel before it (the
    // residual update, or the queue that count_dev counts): every block waits
    // for it before reading the residuals, the count or the keys, then lets
    // the next kernel launch
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    constexpr int kWarps = kGemvThreads / 32;
    const int64_t gw = (int64_t)blockIdx.x * kWarps + wid;
    const int64_t nw = (int64_t)gridDim.x * kWarps;
    const int count = count_dev ? *(const volatile int *)count_dev : B;  // not before the wait
    const int Lp4 = Lp >> 2;
    const float4 *D4 = reinterpret_cast<const float4 *>(D);

    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        fence_mbar_init();
    }
    __syncthreads();
    uint32_t parity = 0;

    for (int g = 0; g < count; ++g) {
        const int ch = chlist ? chlist[g] : g;
        if (threadIdx.x == 0) {
            mbar_expect_tx(&bar, (uint32_t)(Lp * 4));
            bulk_g2s(smem_r, R + (int64_t)ch * Lp, (uint32_t)(Lp * 4), &bar);
        }
        const int timed_out = mbar_wait(&bar, parity, wait_ns) ? 0 : 1;
        if (__syncthreads_or(timed_out)) {
            if (threadIdx.x == 0) {
                atomicOr(status, kFlagTimeout);
                mbar_drain(&bar, parity);  // bounded: let the in-flight copy land before exiting
            }
            return;
        }
        parity ^= 1u;

        float4 rv[NV];
#pragma unroll
        for (int j = 0; j < NV; ++j) rv[j] = reinterpret_cast<const float4 *>(smem_r)[lane + 32 * j];
        float best = -1.0f;
        uint32_t bidx = 0u;
        for (int64_t row = gw; row < K; row += 2 * nw) {
            const int64_t row2 = row + nw;
            const bool has2 = row2 < K;
            float4 a[NV], b[NV];
            const float4 *pa = D4 + row * Lp4 + lane;
#pragma unroll
            for (int j = 0; j < NV; ++j) a[j] = ldg_stream(pa + 32 * j);
            if (has2) {
                const float4 *pb = D4 + row2 * Lp4 + lane;
#pragma unroll
                for (int j = 0; j < NV; ++j) b[j] = ldg_stream(pb + 32 * j);
            } else {
#pragma unroll
                for (int j = 0; j < NV; ++j) b[j] = make_float4(0.f, 0.f, 0.f, 0.f);
            }
            float x0 = 0.f, x1 = 0.f, y0 = 0.f, y1 = 0.f;
#pragma unroll
            for (int j = 0; j < NV; ++j) {
                x0 = fmaf(a[j].x, rv[j].x, x0);
                x1 = fmaf(a[j].y, rv[j].y, x1);
                x0 = fmaf(a[j].z, rv[j].z, x0);
                x1 = fmaf(a[j].w, rv[j].w, x1);
                y0 = fmaf(b[j].x, rv[j].x, y0);
                y1 = fmaf(b[j].y, rv[j].y, y1);
                y0 = fmaf(b[j].z, rv[j].z, y0);
                y1 = fmaf(b[j].w, rv[j].w, y1);
            }
            float sa = x0 + x1, sb = y0 + y1;
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) {
                sa += __shfl_xor_sync(0xffffffffu, sa, off);
                sb += __shfl_xor_sync(0xffffffffu, sb, off);
            }
            if (WRITE) {
                if (lane == 0) {
                    // Looked up at each row: with the channel held from outside
                    // the loop, or left out, ptxas takes 4 to 14 registers less
                    // and a call is slower (Lp 256, 94 MB: 20.7 us, 23.0 and
                    // 26.7 the other ways; Lp 384, 170 MB: 32.9 and 34.8).
                    const int cw = chlist ? chlist[g] : g;
                    scores[(int64_t)cw * K + row] = sa;
                    if (has2) scores[(int64_t)cw * K + row2] = sb;
                }
            } else {
                float x = fabsf(sa);
                if (x > best) {
                    best = x;
                    bidx = (uint32_t)row;
                }
                if (has2) {
                    x = fabsf(sb);
                    if (x > best) {
                        best = x;
                        bidx = (uint32_t)row2;
                    }
                }
            }
        }
        if (!WRITE) {
            if (lane == 0) {
                red_s[wid] = best;
                red_i[wid] = bidx;
            }
            __syncthreads();
            if (threadIdx.x == 0) {
                float bs = -1.0f;
                uint32_t bi = 0u;
                for (int w = 0; w < kWarps; ++w) {
                    const float s = red_s[w];
                    const uint32_t i = red_i[w];
                    if (s > bs || (s == bs && i < bi)) {
                        bs = s;
                        bi = i;
                    }
                }
                if (bs >= 0.0f) atomicMax(keys + ch, pack_key(bs, bi));
            }
        }
        __syncthreads();  // the shared residual and reduction slots are reused by the next channel
    }
}

template <int NV>
static cudaError_t gemv_instance(const float *D, int64_t K, int Lp, const float *R, int B, const int *chlist,
                                 const int *count_dev, unsigned long long *keys, float *scores, int *status,
                                 int grid_ctas, unsigned long long wait_ns, cudaStream_t st, bool pdl) {
    return launch_kernel(scores ? k_gemv<NV, true> : k_gemv<NV, false>, dim3(grid_ctas), dim3(kGemvThreads),
                         (size_t)Lp * sizeof(float), st, pdl, D, K, Lp, R, B, chlist, count_dev, keys, scores, status,
                         wait_ns);
}

int gemv_ctas(int sm_count, int Lp) { return sm_count * gemv_max_ctas_per_sm(Lp); }

int gemv_max_ctas_per_sm(int Lp) {
    int per_sm = 0;
    const int nv = Lp / 128;
    cudaError_t e = cudaErrorInvalidValue;
    const size_t smem = (size_t)Lp * sizeof(float);
    switch (nv) {
        case 1: e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_gemv<1, false>, kGemvThreads, smem); break;
        case 2: e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_gemv<2, false>, kGemvThreads, smem); break;
        case 3: e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_gemv<3, false>, kGemvThreads, smem); break;
        case 4: e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_gemv<4, false>, kGemvThreads, smem); break;
        case 8: e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_gemv<8, false>, kGemvThreads, smem); break;
        case 16: e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_gemv<16, false>, kGemvThreads, smem); break;
        default: break;
    }
    if (e != cudaSuccess || per_sm < 1) per_sm = 1;
    if (per_sm > 4) per_sm = 4;
    return per_sm;
}

static cudaError_t launch_gemv(const float *D, int64_t K, int Lp, const float *R, int B, const int *chlist,
                               const int *count_dev, unsigned long long *keys, float *scores, int *status,
                               int grid_ctas, cudaStream_t st, unsigned long long wait_ns, bool pdl) {
#define ACT_GEMV_CASE(NVV)                                                                                        \
    case NVV:                                                                                                     \
        return gemv_instance<NVV>(D, K, Lp, R, B, chlist, count_dev, keys, scores, status, grid_ctas, wait_ns, st, \
                                  pdl);
    switch (Lp / 128) {
        ACT_GEMV_CASE(1)
        ACT_GEMV_CASE(2)
        ACT_GEMV_CASE(3)
        ACT_GEMV_CASE(4)
        ACT_GEMV_CASE(8)
        ACT_GEMV_CASE(16)
        default:
            return cudaErrorInvalidValue;
    }
#undef ACT_GEMV_CASE
}

cudaError_t launch_gemv_argmax(const float *D, int64_t K, int Lp, const float *R, int B, const int *chlist,
                               const int *count_dev, unsigned long long *keys, int *status, int grid_ctas,
                               cudaStream_t st, unsigned long long wait_ns, bool pdl) {
    return launch_gemv(D, K, Lp, R, B, chlist, count_dev, keys, nullptr, status, grid_ctas, st, wait_ns, pdl);
}

cudaError_t launch_gemv_scores(const float *D, int64_t K, int Lp, const float *R, int B, float *scores, int *status,
                               int grid_ctas, cudaStream_t st, unsigned long long wait_ns) {
    return launch_gemv(D, K, Lp, R, B, nullptr, nullptr, nullptr, scores, status, grid_ctas, st, wait_ns, false);
}

}  // namespace act
