// FP32 search and projection of several channels over the stored dictionary,
// up to 16 channels per pass over it.  With one score per (row, channel) the
// butterfly sum alone takes five shuffles and five adds, more than the row's
// multiplies at N = 512; here a warp scores a tile of 8 rows x 4 or 8
// channels and reduces 32 sums together: at every step of the butterfly a
// lane keeps half of its sums and sends the other half, 31 shuffles for 32
// scores, each lane left with one.  The additions are the butterfly's own
// (the two operands exchanged at most), and a row's products are added in
// the GEMV's order, so every score has the GEMV's bits.  The dictionary
// streams through shared memory by TMA bulk copies (as in k_gemv_stream) and
// is read once per 16 channels: bound by HBM from 4 GB dictionaries on (four
// channels' scores of 2,097,152 x 512 atoms: 1,242 us in passes of 4, now 650
// = 6.7 TB/s), by issue and by the shared-memory reads of rows and residuals
// in L2-resident ones (12 channels of 113,778 x 256 atoms: 100 us an order in
// passes of 4, now 44; 53 with the 12 padded to 16).
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "act_device.cuh"
#include "act_internal.cuh"

namespace act {

namespace {

// consumers: with the producer two warps a scheduler, 255 registers a thread
constexpr int kMultiWarps = 7;
constexpr int kMultiThreads = (kMultiWarps + 1) * 32;   // + the producer
constexpr int kTileRows = 8;
constexpr int kMultiMaxStages = 12;
constexpr int kMultiChannels = 16;        // per pass
constexpr int kMultiRing = 196608;        // bytes of the stages
constexpr int kMultiResid = 32768;        // bytes of a pass's residuals
constexpr int kMultiChunk = 32768;        // bytes of a stage, where a tile is not larger

__device__ __forceinline__ unsigned long long pair_of(float a, float b) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void fma_pair(unsigned long long &acc, unsigned long long a, unsigned long long b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}
__device__ __forceinline__ float pair_sum(unsigned long long v) {
    float a, b;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
    return a + b;
}

// Sums of 32 values over the warp: lane l returns the total of v[l].
__device__ __forceinline__ float warp_sum_32(float (&v)[32], int lane) {
#pragma unroll
    for (int half = 16; half > 0; half >>= 1) {
        const bool up = (lane & half) != 0;
#pragma unroll
        for (int i = 0; i < half; ++i) {
            const float send = up ? v[i] : v[i + half];
            const float keep = up ? v[i + half] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, half);
        }
    }
    return v[0];
}

// N8 groups of 8 channels and N4 of 4 (ng <= 8 N8 + 4 N4 channels in all; the
// residuals of the missing ones are zero).  A chunk is `tiles` tiles of 8
// rows, tile t of this CTA's i-th chunk for warp (i tiles + t) mod 7.  Every
// consumer warp waits for and releases every chunk, its own tiles or not: a
// warp that skipped chunks could look at a stage two uses ahead while an
// older copy is still in flight, and a parity wait would let it pass.
template <int N8, int N4, bool WRITE_SCORES>
__global__ void __launch_bounds__(kMultiThreads, 1)
    k_gemv_multi(const float *__restrict__ D, int64_t K, int Lp, const float *R, int ng,
                 unsigned long long *keys, float *scores, int tiles, int stages, int *status,
                 unsigned long long wait_ns) {
    constexpr int NCH = 8 * N8 + 4 * N4, G = N8 + N4;
    extern __shared__ __align__(128) float sm[];  // stages, then [NCH][Lp] residuals
    __shared__ __align__(8) uint64_t full[kMultiMaxStages], empty[kMultiMaxStages];
    __shared__ float red_s[kMultiWarps][NCH];
    __shared__ uint32_t red_i[kMultiWarps][NCH];
    __shared__ int abort_sh;
    __shared__ unsigned long long issued_sh;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int rows_per_chunk = tiles * kTileRows;
    const int64_t total_chunks = (K + rows_per_chunk - 1) / rows_per_chunk;
    const int64_t n_chunks = total_chunks > blockIdx.x ? (total_chunks - blockIdx.x + gridDim.x - 1) / gridDim.x : 0;
    const size_t stage_floats = (size_t)rows_per_chunk * Lp;
    float *res = sm + stages * stage_floats;
    if (threadIdx.x == 0) {
        for (int s = 0; s < stages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], kMultiWarps);
        }
        abort_sh = 0;
        issued_sh = 0ull;
        fence_mbar_init();
    }
    __syncthreads();
    // The dictionary is constant: its first chunks are on their way before
    // the kernel before this one (the residual update) is waited for.
    auto issue = [&](int64_t k) {  // the producer's one thread
        const int s = (int)(k % stages);
        const int64_t row = (blockIdx.x + k * gridDim.x) * rows_per_chunk;
        const int64_t nrows = K - row < rows_per_chunk ? K - row : rows_per_chunk;
        const uint32_t bytes = (uint32_t)(nrows * Lp * 4);
        mbar_expect_tx(&full[s], bytes);
        bulk_g2s(sm + s * stage_floats, D + row * Lp, bytes, &full[s]);
        *(volatile unsigned long long *)&issued_sh = (unsigned long long)k + 1ull;
    };
    const bool producer = wid == kMultiWarps;
    int64_t first = 0;
    if (producer && lane == 0)
        for (; first < n_chunks && first < stages; ++first) issue(first);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    for (int i = threadIdx.x; i < NCH * Lp; i += kMultiThreads) res[i] = i < ng * Lp ? R[i] : 0.0f;
    __syncthreads();

    if (producer) {
        if (lane == 0) {
            for (int64_t k = first; k < n_chunks; ++k) {
                if (!mbar_wait(&empty[k % stages], (uint32_t)((k / stages) & 1) ^ 1u, wait_ns)) {
                    abort_sh = 1;
                    break;
                }
                issue(k);
            }
        }
    } else {
        float best[NCH / 4];  // lane: row (lane & 7) of a tile, channel 4 h + (lane >> 3)
        uint32_t bidx[NCH / 4];
#pragma unroll
        for (int h = 0; h < NCH / 4; ++h) {
            best[h] = -1.0f;
            bidx[h] = 0u;
        }
        const int nv = Lp >> 7;
        int s = 0, off = 0;  // the stage, and the warp of the chunk's first tile
        uint32_t ph = 0u;
        for (int64_t k = 0; k < n_chunks; ++k) {
            const int ok = mbar_wait(&full[s], ph, wait_ns) ? 1 : 0;
            if (!__all_sync(0xffffffffu, ok)) {
                if (lane == 0) abort_sh = 1;
                break;
            }
            int t = wid - off;
            t = t < 0 ? t + kMultiWarps : t;
            if (t >= tiles) {  // none of this chunk's tiles is this warp's
                if (lane == 0) mbar_arrive(&empty[s]);
            }
            for (; t < tiles; t += kMultiWarps) {
                const int64_t row0 = ((int64_t)blockIdx.x + k * gridDim.x) * rows_per_chunk + t * kTileRows;
                const float4 *a4 =
                    reinterpret_cast<const float4 *>(sm + s * stage_floats + (size_t)t * kTileRows * Lp) + lane;
                const int ld = Lp >> 2;
                // one group of NB channels from c0 on; `last`: the warp's last read of the stage
                auto group = [&](auto nb, int c0, bool last) {
                    constexpr int NB = decltype(nb)::value;
                    unsigned long long acc[NB][kTileRows];
#pragma unroll
                    for (int c = 0; c < NB; ++c)
#pragma unroll
                        for (int r = 0; r < kTileRows; ++r) acc[c][r] = 0ull;
                    const float4 *r4 = reinterpret_cast<const float4 *>(res + (size_t)c0 * Lp) + lane;
#pragma unroll 1
                    for (int j = 0; j < nv; ++j) {
                        unsigned long long xy[kTileRows], zw[kTileRows];
#pragma unroll
                        for (int r = 0; r < kTileRows; ++r) {
                            const float4 a = a4[r * ld + 32 * j];
                            xy[r] = pair_of(a.x, a.y);
                            zw[r] = pair_of(a.z, a.w);
                        }
#pragma unroll
                        for (int c = 0; c < NB; ++c) {
                            const float4 v = r4[c * ld + 32 * j];
                            const unsigned long long vxy = pair_of(v.x, v.y), vzw = pair_of(v.z, v.w);
#pragma unroll
                            for (int r = 0; r < kTileRows; ++r) {
                                fma_pair(acc[c][r], xy[r], vxy);
                                fma_pair(acc[c][r], zw[r], vzw);
                            }
                        }
                    }
                    if (last) {
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&empty[s]);
                    }
                    const int64_t row = row0 + (lane & 7);
#pragma unroll
                    for (int q = 0; q < NB / 4; ++q) {
                        float v[32];
#pragma unroll
                        for (int i = 0; i < 32; ++i) v[i] = pair_sum(acc[q * 4 + (i >> 3)][i & 7]);
                        const float sc = warp_sum_32(v, lane);
                        if (row < K) {
                            if (WRITE_SCORES) {
                                const int c = c0 + q * 4 + (lane >> 3);
                                if (c < ng) scores[(int64_t)c * K + row] = sc;
                            } else {
                                const float x = fabsf(sc);
                                if (x > best[c0 / 4 + q]) {  // a lane's rows ascend: the first of equal scores stays
                                    best[c0 / 4 + q] = x;
                                    bidx[c0 / 4 + q] = (uint32_t)row;
                                }
                            }
                        }
                    }
                };
                const bool end = t + kMultiWarps >= tiles;  // this warp's last tile of the chunk
#pragma unroll
                for (int g = 0; g < N8; ++g) group(std::integral_constant<int, 8>(), 8 * g, end && g == G - 1);
                if constexpr (N4 > 0) group(std::integral_constant<int, 4>(), 8 * N8, end);
            }
            off += tiles;
            while (off >= kMultiWarps) off -= kMultiWarps;
            if (++s == stages) {
                s = 0;
                ph ^= 1u;
            }
        }
        if (!WRITE_SCORES) {
#pragma unroll
            for (int h = 0; h < NCH / 4; ++h) {
                float bs = best[h];
                uint32_t bi = bidx[h];
                for (int o = 4; o > 0; o >>= 1) {
                    const float os = __shfl_xor_sync(0xffffffffu, bs, o);
                    const uint32_t oi = __shfl_xor_sync(0xffffffffu, bi, o);
                    if (os > bs || (os == bs && oi < bi)) {
                        bs = os;
                        bi = oi;
                    }
                }
                if ((lane & 7) == 0) {
                    red_s[wid][4 * h + (lane >> 3)] = bs;
                    red_i[wid][4 * h + (lane >> 3)] = bi;
                }
            }
        }
    }
    __syncthreads();
    if (abort_sh) {
        if (threadIdx.x == 0) {
            atomicOr(status, kFlagTimeout);
            // let every copy in flight land before the CTA exits: stage s took
            // issue numbers s, s + stages, ...; wait for the phase of its last
            const unsigned long long n = issued_sh;
            for (int s = 0; s < stages; ++s)
                if (n > (unsigned long long)s)
                    mbar_drain(&full[s], (uint32_t)(((n - 1 - s) / (unsigned long long)stages) & 1ull));
        }
        return;
    }
    if (!WRITE_SCORES && threadIdx.x < ng) {
        const int c = threadIdx.x;
        float bs = -1.0f;
        uint32_t bi = 0u;
        for (int w = 0; w < kMultiWarps; ++w)
            if (red_s[w][c] > bs || (red_s[w][c] == bs && red_i[w][c] < bi)) {
                bs = red_s[w][c];
                bi = red_i[w][c];
            }
        if (bs >= 0.0f) atomicMax(keys + c, pack_key(bs, bi));
    }
}

template <int N8, int N4, bool WS>
cudaError_t multi_instance(const float *D, int64_t K, int Lp, const float *R, int ng, unsigned long long *keys,
                           float *scores, int *status, int sm_count, cudaStream_t st, unsigned long long wait_ns,
                           bool pdl) {
    // Tiles per chunk, at most 32 KB of them: the fewest that give no CTA a
    // second chunk where that can be (a warp's first tile is then its only one
    // in most), else a power of two that leaves every SM two chunks.  us per
    // order, 4 channels, rows of 128 floats: 2 MB 6.84 by the second rule
    // alone and 6.15, 4 MB 8.12 and 6.67 (the GEMV in passes of four channels
    // took 7.3), of 256 floats: 8 MB 7.80 and 7.12.
    const int64_t total = (K + kTileRows - 1) / kTileRows;
    int most = 1;
    while (2 * most * kTileRows * Lp * 4 <= kMultiChunk) most *= 2;
    int tiles = (int)(total <= (int64_t)most * sm_count ? (total + sm_count - 1) / sm_count : most);
    if (total > (int64_t)most * sm_count)
        while (tiles > 1 && (K + tiles * kTileRows - 1) / (tiles * kTileRows) < 2 * (int64_t)sm_count) tiles /= 2;
    const int chunk = tiles * kTileRows * Lp * 4;
    int stages = kMultiRing / chunk;
    if (stages > kMultiMaxStages) stages = kMultiMaxStages;
    const size_t smem = (size_t)stages * chunk + sizeof(float) * (size_t)(8 * N8 + 4 * N4) * Lp;
    // set for the current device on every launch; no allocation, legal in a capture
    cudaError_t e = cudaFuncSetAttribute(k_gemv_multi<N8, N4, WS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         kMultiRing + kMultiResid);
    if (e != cudaSuccess) return e;
    const int64_t chunks = (K + tiles * kTileRows - 1) / (tiles * kTileRows);
    return launch_kernel(k_gemv_multi<N8, N4, WS>, dim3((unsigned)(chunks < sm_count ? chunks : sm_count)),
                         dim3(kMultiThreads), smem, st, pdl, D, K, Lp, R, ng, keys, scores, tiles, stages, status,
                         wait_ns);
}

template <bool WS>
cudaError_t multi_passes(const float *D, int64_t K, int Lp, const float *R, int B, unsigned long long *keys,
                         float *scores, int *status, int sm_count, cudaStream_t st, unsigned long long wait_ns,
                         bool pdl) {
    // channels per pass: what the residuals' shared memory holds, at most 16
    int most = kMultiResid / (Lp * 4);
    most = most >= kMultiChannels ? kMultiChannels : (most >= 8 ? 8 : 4);
    for (int c0 = 0; c0 < B; c0 += most) {
        const int ng = B - c0 < most ? B - c0 : most;
        const float *r = R + (size_t)c0 * Lp;
        unsigned long long *k = WS ? nullptr : keys + c0;
        float *sc = WS ? scores + (int64_t)c0 * K : nullptr;
        cudaError_t e;
#define ACT_MULTI(N8, N4) multi_instance<N8, N4, WS>(D, K, Lp, r, ng, k, sc, status, sm_count, st, wait_ns, pdl)
        e = ng <= 4 ? ACT_MULTI(0, 1) : ng <= 8 ? ACT_MULTI(1, 0) : ng <= 12 ? ACT_MULTI(1, 1) : ACT_MULTI(2, 0);
#undef ACT_MULTI
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace

cudaError_t launch_gemv_multi_argmax(const float *D, int64_t K, int Lp, const float *R, int B,
                                     unsigned long long *keys, int *status, int sm_count, cudaStream_t st,
                                     unsigned long long wait_ns, bool pdl) {
    return multi_passes<false>(D, K, Lp, R, B, keys, nullptr, status, sm_count, st, wait_ns, pdl);
}

cudaError_t launch_project(const float *D, int64_t K, int Lp, const float *R, int B, float *scores, int *status,
                           int sm_count, int gemv_grid, cudaStream_t st, unsigned long long wait_ns) {
    if (B == 1 ? K * (int64_t)Lp * (int64_t)sizeof(float) < project_multi_bytes(Lp) : one_by_one(K, Lp, B))
        return launch_gemv_scores(D, K, Lp, R, B, scores, status, gemv_grid, st, wait_ns);
    return multi_passes<true>(D, K, Lp, R, B, nullptr, scores, status, sm_count, st, wait_ns, false);
}

}  // namespace act
