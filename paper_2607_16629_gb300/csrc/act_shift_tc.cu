// Tensor-core search over the template dictionary, exact with respect to the
// FP32 template search (act_shift.cu):
//  1. the residuals are laid out as shifted rows X[(b, j)][kk] =
//     bf16(r_b[m_lo + kk + tc_j]) (zero outside the window), so that
//     <r_b, u_{t, tc_j}> = sum_kk u_t(m_lo + kk) X[(b, j)][kk]: one GEMM of
//     the BF16 templates (N = 256 templates per tile) against the shifted
//     residual rows (M = 128 rows per tile), K = Kt lags.  A tile multiplies
//     only the lags that its rows' windows see and its templates span
//     (k_shift_spans): the GEMM is bounded by the tensor pipe and the issue of
//     its MMAs, so fewer lags is what helps (multiplying every lag the windows
//     see, 256 uneven EMG-like channels, atoms of 9-111 samples in windows of
//     256-2,048, took 57.8 ms per 30-order decomposition, now 21.2; 32
//     radar-like channels 4.54 and 3.65, 64 EEG-like channels 2.40 and 1.74);
//  2. the tcgen05 GEMM scales every accumulator by its atom's 1/|u| and keeps,
//     per row, the largest |score| of every template tile and of every
//     32-template block;
//  3. a flag kernel bounds the BF16 error per channel and flags the
//     (time centre, 32-template block) items that can hold the FP32 template
//     search's argmax (scanning the tile maxima, then the flagged tiles' blocks);
//  4. the flagged items are rescored with the FP32 template search's own
//     arithmetic (same FMA chain, same scale) and folded into the packed key;
//     a channel with too many items has all of its items rescored that way.
// Steps 3 and 4 make the selection bit-identical to the FP32 template search.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <new>

#include "act_device.cuh"
#include "act_internal.cuh"
#include "act_tc.cuh"

namespace act {

namespace {

using namespace tc;

// (a0 b0, a1 b1) by one packed FP32 multiply, each product rounded to
// nearest as a scalar multiply would be: the epilogue shares its warp
// scheduler with the MMA-issuing warp, so its instruction count matters.
__device__ __forceinline__ float2 mul_f32x2(float a0, float a1, float b0, float b1) {
    unsigned long long x, y, r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(x) : "f"(a0), "f"(a1));
    asm("mov.b64 %0, {%1, %2};" : "=l"(y) : "f"(b0), "f"(b1));
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(x), "l"(y));
    float2 o;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(o.x), "=f"(o.y) : "l"(r));
    return o;
}

// Bounded wait on a phase by polling test_wait (never suspending the
// thread), with an optional pause between polls; PAIR: cluster-scope
// acquire.  The MMA-issuing thread polls without pausing, so it resumes the
// moment a stage lands; the epilogue pauses, taking fewer issue slots from
// the MMA-issuing warp that shares its scheduler.  Limit 0: one test.
template <bool PAIR>
__device__ __forceinline__ bool mbar_poll(uint64_t *bar, uint32_t parity, unsigned long long limit_ns,
                                          unsigned pause_ns) {
    auto test = [&]() { return PAIR ? mbar_test_wait_cluster(bar, parity) : mbar_test_wait(bar, parity); };
    if (test()) return true;
    if (limit_ns == 0) return false;
    const unsigned long long t0 = globaltimer_ns();
    while (!test()) {
        if (globaltimer_ns() - t0 >= limit_ns) return false;
        if (pause_ns) __nanosleep(pause_ns);
    }
    return true;
}

constexpr int kBM = 128;          // shifted residual rows per tile (MMA M)
constexpr int kBlockRows = 256;   // templates per block of the tile-major BF16 layout
constexpr int kUmmaK = 16;
constexpr int kStepsPerChunk = kBK / kUmmaK;
constexpr int kMaxThreads = 384;  // two epilogue groups
constexpr int kAChunkBytes = kBM * kBK * 2;  // 16 KB
constexpr int kMaxStages = 6;
constexpr unsigned kAccPause = 64;  // ns between an epilogue group's looks at its accumulator
constexpr int kUnitTab = 1024;  // row units whose lag range is tabulated in shared memory
constexpr int kTileTab = 512;   // template tiles whose lag span is

// Tile of BN templates (128 or 256, MMA N).  PAIR: a CTA pair shares each
// MMA (M = 256: the two CTAs' row tiles), each CTA loading BN / 2 of the
// templates; every CTA still holds a 128 x BN accumulator of its own rows.
template <int BN, bool PAIR = false>
struct ShiftTile {
    static constexpr int kBRows = PAIR ? BN / 2 : BN;  // template rows this CTA loads
    static constexpr int kBChunkBytes = kBRows * kBK * 2;
    static constexpr int kStageBytes = kAChunkBytes + kBChunkBytes;
    static constexpr uint32_t kTmemCols = 2 * BN;
    static constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) |
                                       ((uint32_t)((PAIR ? 2 * kBM : kBM) >> 4) << 24);
};
constexpr int kMaxItems = 1024;    // flagged (lag, block) items per channel before the full FP32 search
constexpr int kMaxRowItems = 512;  // the same where the items are rows of a stored dictionary
constexpr int kRescanWarps = 4;     // independent warps per rescore block
constexpr int kRescanBufs = 8;      // phase buffers per warp, at most
// Bytes of a warp's residual and buffers where it has more than two: with few
// channels (few items) one or two warps an SM with every phase in flight, with
// many four warps an SM.  One EEG-like channel 511 us per decomposition and 536
// with two buffers a warp, 64 of them 1,768 with four and 1,730 with two.
// Where not every phase has a buffer there is little to gain and warps to
// lose: EMG-like channels of 2,048 samples, 30 orders, three buffers and two,
// 1 channel 1.414 and 1.419 ms, 4 1.796 and 1.798, 8 2.14 and 2.12, 16 2.87
// and 2.69.
constexpr int kRescanFewBytes = 108 * 1024;
constexpr int kRescanFewChannels = 16, kRescanFewPhased = 4;

struct Smem {
    uint64_t bar_full[kMaxStages];
    uint64_t bar_empty[kMaxStages];
    uint64_t bar_acc_full[2];
    uint64_t bar_acc_empty[2];
    uint32_t tmem_base;
    int abort;
    unsigned int chan_max[2][kBM];  // per epilogue group: the tile's channel maxima (float bits)
    // the lag range [x, y] (16-lag steps) of row units 0 .. kUnitTab - 1 and
    // of template tiles 0 .. kTileTab - 1, formed during set-up: the single
    // thread that issues the MMAs reads them at every item instead of
    // dividing (past the tables: computed there)
    short2 unit_steps[kUnitTab];
    short2 tile_steps[kTileTab];
};

// Named barrier `id` over the 128 threads of one epilogue group, returning
// whether any of them passed a nonzero predicate (all of them get the same
// answer).
__device__ __forceinline__ int epilogue_bar_or(int id, int pred) {
    int r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.s32 p, %1, 0;\n\t"
        "bar.red.or.pred q, %2, 128, p;\n\t"
        "selp.s32 %0, 1, 0, q;\n\t}"
        : "=r"(r)
        : "r"(pred), "r"(id)
        : "memory");
    return r;
}
__device__ __forceinline__ void epilogue_bar(int id) { asm volatile("bar.sync %0, 128;" ::"r"(id) : "memory"); }

// max(|a|, |b|, |c|) in one instruction; a NaN operand is passed over, as fmaxf does.
__device__ __forceinline__ float max_abs3(float a, float b, float c) {
    float r;
    asm("max.abs.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// Row tiles of the GEMM: tile mt = g * n_cb + cb holds Bg = 128 / Jt
// channels (cb * Bg ..) times Jt neighbouring time centres (g * Jt ..); local
// row lr = (j - g Jt) Bg + (b - cb Bg), channels fastest, so with Bg >= 32
// the 32 rows an epilogue warp holds share one time centre (its scale loads
// are broadcasts).  Rows of one tile see the window only over
// L + (Jt - 1) S lags instead of Kt; outside them every product is zero.
// A few channels past the whole blocks have tiles of their own behind the
// others, from m_main on: Bg2 channels (B_main ..) x Jt2 time centres
// (make_tiling).
struct RowTiling {
    int B, Ntc, Jt, Bg, n_cb, m_tiles;
    int S, L, span0;  // span0 = -m_lo - tc0 = S (Ntc - 1); sample n at time centre j sits at lag n + span0 - S j
    int m_main, B_main, Jt2, Bg2;
};

// Row tile mt: channels b0 .. b0 + Bg - 1, time centres j0 .. j0 + Jt - 1.
struct TileGeo {
    int Bg, Jt, b0, j0;
};
__host__ __device__ inline TileGeo tile_geo(const RowTiling &t, int mt) {
    if (t.Jt2 > 0 && mt >= t.m_main) return {t.Bg2, t.Jt2, t.B_main, (mt - t.m_main) * t.Jt2};
    const int g = mt / t.n_cb;
    return {t.Bg, t.Jt, (mt - g * t.n_cb) * t.Bg, g * t.Jt};
}

// The lags row tile mt's windows see, in steps of 16 (one MMA).
__host__ __device__ inline void row_steps(const RowTiling &t, int mt, int &lo, int &hi) {
    const TileGeo geo = tile_geo(t, mt);
    const int j_first = geo.j0;
    const int j_last = min(j_first + geo.Jt, t.Ntc) - 1;
    const int kk_min = t.span0 - t.S * j_last;           // sample 0 at the last time centre
    const int kk_max = t.L - 1 + t.span0 - t.S * j_first;  // sample L - 1 at the first
    lo = kk_min / kUmmaK;
    hi = kk_max / kUmmaK;
}

// Lags of GEMM row unit u: one row tile, or (pair) the union of row tiles 2u
// and 2u + 1 (the second clamped to the last tile).
__host__ __device__ inline short2 unit_steps(const RowTiling &t, bool pair, int u) {
    int lo, hi;
    if (!pair) {
        row_steps(t, u, lo, hi);
    } else {
        int lo1, hi1;
        row_steps(t, 2 * u, lo, hi);
        row_steps(t, min(2 * u + 1, t.m_tiles - 1), lo1, hi1);
        lo = min(lo, lo1);
        hi = max(hi, hi1);
    }
    return make_short2((short)lo, (short)hi);
}

// Lags template tile nt of BN templates spans (k_shift_spans).
template <int BN>
__device__ __forceinline__ short2 tile_steps(const short2 *__restrict__ span, int nt) {
    short2 s = span[nt * (BN / 128)];
    if (BN == 256) {
        const short2 s1 = span[nt * 2 + 1];
        s.x = min(s.x, s1.x);
        s.y = max(s.y, s1.y);
    }
    return s;
}

// The steps an item multiplies: those its rows see and its templates span.
// An empty intersection (only atoms without energy) takes the rows' first
// step, so that the accumulator is written.
__device__ __forceinline__ void item_steps(short2 rows, short2 tpls, int &lo, int &hi) {
    lo = max((int)rows.x, (int)tpls.x);
    hi = min((int)rows.y, (int)tpls.y);
    if (lo > hi) lo = hi = rows.x;
}

// Shifted residual rows X[(b, j)][kk] = bf16(r_b[m_lo + kk + tc0 + S j]),
// zero where the index leaves [0, L).  Block (g * n_seg + seg, b) writes
// channel b's rows for time centres j0 = g RJ .. j0 + RJ - 1 (those below
// Ntc), lags kk in [k0, k1) = [seg KSEG, min(Kt, (seg + 1) KSEG)).  It stages
// the samples those pieces cover, n_lo + i for i in [0, span) with
// n_lo = m_lo + tc0 + S j0 + k0 and span = S (rows - 1) + k1 - k0, as BF16
// in shared memory: once as read (global loads issued four at a time), then
// in 8 copies shifted by 0..7 samples built from it (copy s holds sample
// i + s at i): the 8 samples of any 16-byte output piece, at offset
// o = S jj + kk - k0, are one aligned 16-byte load from copy o & 7.  Padding
// rows (b >= B or j >= Ntc) are not written (the GEMM's epilogue ignores
// them).  Block (0, b) also prepares channel b's selection for this order:
// the error bound of its scores (k_shift_flag), the channel maximum and item
// count cleared.  The bound is formed here because its residual sums are, and
// its FP64 steps take a warp that few channels leave without rows; the flag
// kernel reads it, as all that earlier kernels write, behind its own wait.
//
// With s the exact score, f the FP32 search's score and h the tensor-core
// score of an atom,
//   |f - s| <= eps_r = err_terms 2^-23 |r|
// (template search: one FP32 chain of L products, the FP32 scale and the
// final product; a stored row: the GEMV's sum and the row's own two
// roundings), and
//   |h - s| <= delta = (1 + 1e-5) [eps_u (|r| + |dr|) + |dr|
//                                  + Kt 2^-23 (1 + eps_u)(|r| + |dr|)]
// (eps_u = largest |u~ - u| / |u| over the atoms' windows, u~ = the BF16
// template as multiplied, zero outside its tile's span; dr =
// bf16(r) - r, the Kt term bounds FP32 accumulation in the tensor core, the
// factor the scale product).  bound = 2 delta + 2 eps_r, rounded up.
__global__ void __launch_bounds__(256) k_shift_rows(RowTiling t, const float *R, int Lp, int tc0,
                                                    int m_lo, int Kt, int RJ, int KSEG, int n_seg, int span_pad,
                                                    int err_terms, const unsigned int *__restrict__ eps_bits,
                                                    __nv_bfloat16 *X, float *bound, unsigned int *chmax,
                                                    int *chcount, long long *stats) {
    extern __shared__ __align__(16) uint8_t rows_raw[];
    __shared__ float sh[32];
    // a programmatic dependent of the previous kernel (the residual update):
    // wait for it in every block, then let the GEMM launch
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int b = blockIdx.y, g = blockIdx.x / n_seg, seg = blockIdx.x - g * n_seg;
    const int j0 = g * RJ, nj = min(RJ, t.Ntc - j0);
    const int k0 = seg * KSEG, k1 = min(Kt, k0 + KSEG);
    const int L = t.L, S = t.S;
    const float *r = R + (size_t)b * Lp;
    float te = 0.0f, tde = 0.0f;  // block (0, b): |r|^2 and |bf16(r) - r|^2
    if (blockIdx.x == 0) {
        // FP32 sums of at most 2048 squares are within 2048 * 2^-24 < 1.3e-4
        // (relative) of the exact ones: inflated by 1e-3 they bound them
        float e = 0.0f, de = 0.0f;
        for (int n = threadIdx.x; n < L; n += blockDim.x) {
            const float x = r[n];
            const float d = __bfloat162float(__float2bfloat16_rn(x)) - x;  // exact
            e = fmaf(x, x, e);
            de = fmaf(d, d, de);
        }
        te = block_sum(e, sh);
        tde = block_sum(de, sh);
        if (threadIdx.x == 0) {
            chmax[b] = 0u;
            chcount[b] = 0;
            atomicAdd((unsigned long long *)&stats[0], 1ull);
        }
    }
    if (nj <= 0 || k0 >= k1) return;
    // the 8 shifted BF16 copies, span_pad (a multiple of 8, >= span) samples
    // each, then the plain staged window of span_pad + 8 samples
    __nv_bfloat16 *plain = reinterpret_cast<__nv_bfloat16 *>(rows_raw) + 8 * span_pad;
    const int n_lo = m_lo + tc0 + S * j0 + k0;
    const int total = span_pad + 8;
    for (int i0 = threadIdx.x; i0 < total; i0 += 4 * blockDim.x) {
        float x[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int i = i0 + u * blockDim.x, n = n_lo + i;
            x[u] = (i < total && n >= 0 && n < L) ? r[n] : 0.0f;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int i = i0 + u * blockDim.x;
            if (i < total) plain[i] = __float2bfloat16_rn(x[u]);
        }
    }
    __syncthreads();
    // copy s, pair q = plain samples 2q + s and 2q + s + 1: as 32-bit words of
    // the plain window, word q + s / 2, shifted by a half word when s is odd
    const int half = span_pad >> 1;
    const uint32_t *pw = reinterpret_cast<const uint32_t *>(plain);
    uint32_t *cw = reinterpret_cast<uint32_t *>(rows_raw);
    for (int q = threadIdx.x; q < half; q += blockDim.x) {
        uint32_t w[5];
#pragma unroll
        for (int u = 0; u < 5; ++u) w[u] = pw[q + u];
#pragma unroll
        for (int sft = 0; sft < 8; ++sft)
            cw[sft * half + q] = (sft & 1) ? __funnelshift_r(w[sft >> 1], w[(sft >> 1) + 1], 16) : w[sft >> 1];
    }
    __syncthreads();
    const uint4 *cp16 = reinterpret_cast<const uint4 *>(rows_raw);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // (block (0, b) always gets here: it has rows and lags)
    if (blockIdx.x == 0 && threadIdx.x == blockDim.x - 32) {
        const double rn = sqrt((double)te * (1.0 + 1e-3)), drn = sqrt((double)tde * (1.0 + 1e-3));
        const double eps_u = (double)__uint_as_float(*eps_bits);
        const double rr = rn + drn;
        const double ulp = 1.1920928955078125e-07;  // 2^-23
        const double delta = (1.0 + 1e-5) * (eps_u * rr + drn + (double)Kt * ulp * (1.0 + eps_u) * rr);
        const double eps_r = (double)err_terms * ulp * rn;
        bound[b] = __double2float_ru(2.0 * delta + 2.0 * eps_r);
    }
    const int c0 = k0 >> 3, c1 = k1 >> 3;
    // this channel's tiles: every n_cb-th from first on
    const bool main = b < t.B_main;
    const int Jt = main ? t.Jt : t.Jt2, Bg = main ? t.Bg : t.Bg2, n_cb = main ? t.n_cb : 1;
    const int cb = main ? b / Bg : 0, bl = main ? b - cb * Bg : b - t.B_main, first = main ? cb : t.m_main;
    for (int jj = warp; jj < nj; jj += blockDim.x >> 5) {
        const int j = j0 + jj, gt = j / Jt, jl = j - gt * Jt;
        const int row = (gt * n_cb + first) * kBM + jl * Bg + bl;
        uint4 *out = reinterpret_cast<uint4 *>(X + (size_t)row * Kt);
        for (int c = c0 + lane; c < c1; c += 32) {
            const int o = S * jj + 8 * c - k0, sft = o & 7;
            out[c] = cp16[(sft * span_pad + (o - sft)) >> 3];
        }
    }
}

// GEMM work item w: row unit w / n_tiles, template tile w % n_tiles.  Every
// stage holds one template chunk (BN x 64) and the matching residual chunk
// (128 x 64).  Warp 0: TMA producer; warp 1: MMA issuer; warp 2: tensor
// memory owner; warps 4-7, and 8-11 where launched: epilogue groups (thread =
// residual row).  Two groups take alternate items, one accumulator each: a
// narrow tile's MMAs take less time than one group needs to stage a tile's
// scales, read its accumulator and store its maxima.
//
// PAIR (launched as clusters of 2): a unit is the row tiles 2u and 2u + 1,
// one per CTA of the pair, over the union of their lag chunks.  Each CTA
// loads its rows and its half of the template chunk, both copies counted on
// the leader's (rank 0) full barrier; the leader issues the M = 256 MMAs and
// its commits arrive on both CTAs' barriers; each CTA's epilogue reads its
// own accumulator and releases it on the leader's barrier.
template <int BN, bool PAIR>
__global__ void __launch_bounds__(kMaxThreads, 1)
    k_shift_gemm(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, RowTiling tl,
                 int n_tiles, int nkc, int stages, int T_pad, const short2 *__restrict__ span,
                 const float *__restrict__ scaleT, float *tile_max, float *blk_max, unsigned int *chmax,
                 int *status, unsigned long long wait_ns) {
    // shared memory: stages, then the item's scales [Jt][BN + 4] (the +4
    // floats of padding spread the Jt rows a warp reads over the banks)
    using Cfg = ShiftTile<BN, PAIR>;
    constexpr int kBChunkBytes = Cfg::kBChunkBytes, kStageBytes = Cfg::kStageBytes;
    constexpr uint32_t kTmemCols = Cfg::kTmemCols;
    extern __shared__ uint8_t dyn_raw[];
    __shared__ Smem sm;
    const uint32_t base = (smem_u32(dyn_raw) + 1023u) & ~1023u;
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    // PAIR: rank in the pair, the pair's index and count (1-D clusters of 2)
    const uint32_t rank = PAIR ? cta_rank_in_cluster() : 0u;
    const int64_t unit0 = PAIR ? blockIdx.x / 2 : blockIdx.x;
    const int64_t n_units = PAIR ? gridDim.x / 2 : gridDim.x;
    const int m_units = PAIR ? (tl.m_tiles + 1) / 2 : tl.m_tiles;
    const int64_t items = (int64_t)m_units * n_tiles;
    const int Ntc = tl.Ntc;

    if (threadIdx.x == 0) {
        for (int s = 0; s < stages; ++s) {
            mbar_init(&sm.bar_full[s], 1);
            mbar_init(&sm.bar_empty[s], 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(&sm.bar_acc_full[a], 1);
            // PAIR: one arrival per epilogue warp of either CTA
            mbar_init(&sm.bar_acc_empty[a], PAIR ? 8 : 128);
        }
        sm.abort = 0;
        fence_mbar_init();
    }
    if (threadIdx.x < 2 * kBM) sm.chan_max[threadIdx.x / kBM][threadIdx.x % kBM] = 0u;
    for (int u = threadIdx.x; u < m_units && u < kUnitTab; u += blockDim.x) sm.unit_steps[u] = unit_steps(tl, PAIR, u);
    for (int nt = threadIdx.x; nt < n_tiles && nt < kTileTab; nt += blockDim.x)
        sm.tile_steps[nt] = tile_steps<BN>(span, nt);  // constant since the build
    if (warp == 2) {
        if constexpr (PAIR) {  // the same columns in both CTAs, allocated by one warp of each
            asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                             smem_u32(&sm.tmem_base)),
                         "r"(kTmemCols)
                         : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
        } else {
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                             smem_u32(&sm.tmem_base)),
                         "r"(kTmemCols)
                         : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        }
    }
    tc_fence_before();
    __syncthreads();
    // PAIR: both CTAs' barriers initialised and tensor memory allocated
    // before either copies, commits or arrives across the pair
    if constexpr (PAIR) cluster_barrier();
    tc_fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, sm.tmem_base, 0);
    volatile int *abort_flag = &sm.abort;
    // set-up above overlaps the shifted-row build; everything below reads its
    // rows (and the channel maxima it cleared) only after it completes
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    if (warp == 0 && lane == 0) {
        // ---------------- TMA producer ----------------
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmA)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmB)) : "memory");
        uint32_t s = 0, ph = 0;  // the ring's stage and its phase parity
        for (int64_t w = unit0; w < items && !*abort_flag; w += n_units) {
            const int u = (int)((uint32_t)w / (uint32_t)n_tiles), nt = (int)((uint32_t)w % (uint32_t)n_tiles);
            // this CTA's row tile (PAIR: past the last tile, load the last one again)
            const int mt = PAIR ? min(2 * u + (int)rank, tl.m_tiles - 1) : u;
            int ks_lo, ks_hi;
            item_steps(u < kUnitTab ? sm.unit_steps[u] : unit_steps(tl, PAIR, u),
                       nt < kTileTab ? sm.tile_steps[nt] : tile_steps<BN>(span, nt), ks_lo, ks_hi);
            const int kc_hi = ks_hi / kStepsPerChunk;
            for (int kc = ks_lo / kStepsPerChunk; kc <= kc_hi; ++kc) {
                const bool ok = PAIR ? mbar_wait_cluster(&sm.bar_empty[s], ph ^ 1u, wait_ns)
                                     : mbar_wait(&sm.bar_empty[s], ph ^ 1u, wait_ns);
                if (!ok) {
                    *abort_flag = 1;
                    break;
                }
                const uint32_t b0 = base + (uint32_t)s * kStageBytes;
                // templates: the tile-major layout seen as [blocks * nkc * 256][64]
                const int64_t t0 = (int64_t)nt * BN + (int64_t)rank * Cfg::kBRows;
                const int64_t blk = t0 / kBlockRows, sub = t0 % kBlockRows;
                const int yB = (int)((blk * nkc + kc) * kBlockRows + sub);
                if constexpr (PAIR) {
                    // both CTAs' copies complete on the leader's barrier
                    if (rank == 0) mbar_expect_tx(&sm.bar_full[s], (uint32_t)(2 * kStageBytes));
                    const uint32_t fb = cluster_addr(&sm.bar_full[s], 0);
                    tma_load_2d_pair(b0, &tmB, 0, yB, fb);
                    tma_load_2d_pair(b0 + kBChunkBytes, &tmA, kc * kBK, mt * kBM, fb);
                } else {
                    mbar_expect_tx(&sm.bar_full[s], (uint32_t)kStageBytes);
                    tma_load_2d(b0, &tmB, 0, yB, &sm.bar_full[s]);
                    tma_load_2d(b0 + kBChunkBytes, &tmA, kc * kBK, mt * kBM, &sm.bar_full[s]);
                }
                if (++s == (uint32_t)stages) {
                    s = 0;
                    ph ^= 1u;
                }
            }
        }
    } else if (warp == 1 && rank == 0) {
        // ---------------- MMA issuer (PAIR: the leader only) ----------------
        // The whole warp runs the loop and one elected lane issues: with the
        // control flow and the operands uniform over the warp, the
        // descriptors stay in uniform registers, where the MMA takes them (lane
        // 0 alone in the loop took about 230 cycles to issue each).  What it
        // has to keep up with is one M x 256 x 16 MMA per 128 cycles: an item
        // of 19.7 MMAs (64 EEG-like channels) takes 3,984 cycles, the rest
        // lost between stages of one to four MMAs.
        tc_fence_after();
        const bool issuer = elect_one();
        uint32_t s = 0, ph = 0, local = 0;
        auto test_full = [&](uint32_t st, uint32_t parity) {
            return PAIR ? mbar_test_wait_cluster(&sm.bar_full[st], parity) : mbar_test_wait(&sm.bar_full[st], parity);
        };
        bool landed = false;  // the stage about to be multiplied was seen complete a stage ago
        for (int64_t w = unit0; w < items; w += n_units, ++local) {
            const uint32_t acc = local & 1u, aph = (local >> 1) & 1u;
            int ks_lo, ks_hi;
            const int u = (int)((uint32_t)w / (uint32_t)n_tiles), nt = (int)(w - (int64_t)u * n_tiles);
            item_steps(u < kUnitTab ? sm.unit_steps[u] : unit_steps(tl, PAIR, u),
                       nt < kTileTab ? sm.tile_steps[nt] : tile_steps<BN>(span, nt), ks_lo, ks_hi);
            ks_lo = __shfl_sync(0xffffffffu, ks_lo, 0);
            ks_hi = __shfl_sync(0xffffffffu, ks_hi, 0);
            const bool ok = PAIR ? mbar_wait_cluster(&sm.bar_acc_empty[acc], aph ^ 1u, wait_ns)
                                 : mbar_wait(&sm.bar_acc_empty[acc], aph ^ 1u, wait_ns);
            if (!__all_sync(0xffffffffu, ok && !*abort_flag)) {
                *abort_flag = 1;
                break;
            }
            tc_fence_after();
            const uint32_t d_tmem = tmem + acc * BN;
            const int kc_lo = ks_lo / kStepsPerChunk, kc_hi = ks_hi / kStepsPerChunk;
            bool all = true;
            for (int kc = kc_lo; kc <= kc_hi; ++kc) {
                if (!landed) {
                    all = __all_sync(0xffffffffu, mbar_poll<PAIR>(&sm.bar_full[s], ph, wait_ns, 0));
                    if (!all) break;
                }
                tc_fence_after();
                const uint32_t s1 = s + 1 == (uint32_t)stages ? 0u : s + 1, ph1 = s1 == 0u ? ph ^ 1u : ph;
                // look at the next stage's barrier now: the answer is there when
                // these MMAs are issued (a look afterwards costs some 290
                // cycles, this one 170)
                const bool next = test_full(s1, ph1);
                const uint32_t b0 = base + s * (uint32_t)kStageBytes;
                // only the chunk's steps inside [ks_lo, ks_hi]
                const int k0 = max(ks_lo - kc * kStepsPerChunk, 0);
                const int n = min(ks_hi - kc * kStepsPerChunk, kStepsPerChunk - 1) - k0 + 1;
                const uint64_t bdesc = smem_desc_k(smem_desc(b0), k0);
                const uint64_t adesc = smem_desc_k(smem_desc(b0 + kBChunkBytes), k0);
                if (issuer) {
                    auto mma = [&](int k, bool accum) {
                        const uint64_t da = smem_desc_k(adesc, k), db = smem_desc_k(bdesc, k);
                        if constexpr (PAIR)
                            tc_mma_pair(d_tmem, da, db, Cfg::kIdesc, accum ? 1u : 0u);
                        else
                            tc_mma(d_tmem, da, db, Cfg::kIdesc, accum ? 1u : 0u);
                    };
                    mma(0, kc != kc_lo);
                    if (n == kStepsPerChunk) {
#pragma unroll
                        for (int k = 1; k < kStepsPerChunk; ++k) mma(k, true);
                    } else {
                        if (n > 1) mma(1, true);
                        if (n > 2) mma(2, true);
                    }
                    if constexpr (PAIR)
                        tc_commit_pair(&sm.bar_empty[s], 0x3);
                    else
                        tc_commit(&sm.bar_empty[s]);
                }
                __syncwarp();
                landed = __all_sync(0xffffffffu, next);
                s = s1;
                ph = ph1;
            }
            if (!all) {
                *abort_flag = 1;
                break;
            }
            if (issuer) {
                if constexpr (PAIR)
                    tc_commit_pair(&sm.bar_acc_full[acc], 0x3);
                else
                    tc_commit(&sm.bar_acc_full[acc]);
            }
            __syncwarp();
        }
    } else if (warp >= 4) {
        // ---------------- epilogue: thread = shifted residual row ----------------
        const int eg = (warp - 4) >> 2, q = warp & 3;  // this warp's group; its quarter of the tensor-memory lanes
        const uint32_t n_eg = (blockDim.x - 128) >> 7;
        const int et = threadIdx.x & 127, bar_id = 1 + eg;
        constexpr int kScaleLd = BN + 4;
        float *sc_sm = reinterpret_cast<float *>(dyn_raw + (base - smem_u32(dyn_raw)) + (size_t)stages * kStageBytes) +
                       (size_t)eg * max(tl.Jt, tl.Jt2) * kScaleLd;
        uint32_t local = (uint32_t)eg;
        for (int64_t w = unit0 + eg * n_units; w < items; w += n_eg * n_units, local += n_eg) {
            const int unit = (int)((uint32_t)w / (uint32_t)n_tiles), nt = (int)((uint32_t)w % (uint32_t)n_tiles);
            const int mt = PAIR ? 2 * unit + (int)rank : unit;  // PAIR: may be one past the last tile (no rows)
            // the tile's Jt scale rows (j0 .. j0 + Jt - 1, those below Ntc), BN each
            const TileGeo geo = tile_geo(tl, mt);
            {
                const int j0 = geo.j0;
                const int rows = min(geo.Jt, Ntc - j0);
                const int per_row = BN / 4;  // 16-byte pieces
                for (int i = et; i < rows * per_row; i += 128) {
                    const int rr = i / per_row, cc = i % per_row;
                    const float *src = scaleT + (size_t)(j0 + rr) * T_pad + (size_t)nt * BN + 4 * cc;
                    const uint32_t dst = smem_u32(sc_sm + rr * kScaleLd + 4 * cc);
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
                }
                asm volatile("cp.async.wait_all;" ::: "memory");
                epilogue_bar(bar_id);
            }
            const uint32_t acc = local & 1u, aph = (local >> 1) & 1u;
            const bool landed = mbar_poll<PAIR>(&sm.bar_acc_full[acc], aph, wait_ns, kAccPause);
            const int failed = (*abort_flag || !landed) ? 1 : 0;
            if (epilogue_bar_or(bar_id, failed)) {  // the group's warps leave together
                *abort_flag = 1;
                break;
            }
            tc_fence_after();
            const int lr = q * 32 + lane;
            const int jl = lr / geo.Bg, bl = lr - jl * geo.Bg;
            const int b = geo.b0 + bl, j = geo.j0 + jl;
            const bool valid = mt < tl.m_tiles && b < tl.B && j < Ntc;
            const float4 *sc4 = reinterpret_cast<const float4 *>(sc_sm + (valid ? jl : 0) * kScaleLd);
            // per 32-template block and per tile: the largest scaled |score|
            float *bm = blk_max + ((size_t)(valid ? b : 0) * Ntc + (valid ? j : 0)) * (T_pad / 32) +
                        (size_t)nt * (BN / 32);
            float mx = 0.0f, bmv[BN / 32];
            // the next 32 columns are on their way while these are scaled
            const uint32_t cols = tmem + ((uint32_t)(q * 32) << 16) + acc * BN;
            uint32_t v[2][32];
            tmem_load32(cols, v[0]);
#pragma unroll
            for (int c = 0; c < BN / 32; ++c) {
                tmem_wait32(v[c & 1]);
                if (c + 1 < BN / 32) tmem_load32(cols + (c + 1) * 32, v[(c + 1) & 1]);
                const uint32_t(&x)[32] = v[c & 1];
                float m0 = 0.0f, m1 = 0.0f;
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const float4 s = valid ? sc4[c * 8 + e] : make_float4(0.f, 0.f, 0.f, 0.f);
                    const float2 p01 =
                        mul_f32x2(__uint_as_float(x[4 * e]), __uint_as_float(x[4 * e + 1]), s.x, s.y);
                    const float2 p23 =
                        mul_f32x2(__uint_as_float(x[4 * e + 2]), __uint_as_float(x[4 * e + 3]), s.z, s.w);
                    m0 = max_abs3(m0, p01.x, p01.y);
                    m1 = max_abs3(m1, p23.x, p23.y);
                }
                bmv[c] = fmaxf(m0, m1);
                mx = fmaxf(mx, bmv[c]);
            }
            tc_fence_before();
            if constexpr (PAIR) {  // one arrival per warp, on the leader's barrier
                __syncwarp();
                if (lane == 0) mbar_arrive_remote(cluster_addr(&sm.bar_acc_empty[acc], 0));
            } else {
                mbar_arrive(&sm.bar_acc_empty[acc]);
            }
            if (valid) {  // the row's BN / 32 block maxima are contiguous: 16-byte stores
                float4 *bm4 = reinterpret_cast<float4 *>(bm);
#pragma unroll
                for (int u = 0; u < BN / 128; ++u)
                    bm4[u] = make_float4(bmv[4 * u], bmv[4 * u + 1], bmv[4 * u + 2], bmv[4 * u + 3]);
                tile_max[((size_t)b * Ntc + j) * n_tiles + nt] = mx;
            }
            // channel maximum: non-negative floats order like their bits.  The
            // rows of one channel are the lanes lr % Bg equal: fold them within
            // the warp, then across the warps in shared memory; one global
            // atomic per channel and tile
            unsigned bits = valid ? __float_as_uint(mx) : 0u;
            for (int off = 16; off >= geo.Bg; off >>= 1) {
                const unsigned o = __shfl_xor_sync(0xffffffffu, bits, off);
                bits = o > bits ? o : bits;
            }
            unsigned int *cm = sm.chan_max[eg];
            if (geo.Bg >= 32 || lane < geo.Bg) atomicMax(cm + bl, bits);
            epilogue_bar(bar_id);  // also: the scale rows are reloaded for the next item
            if (et < geo.Bg) {
                const int bc = geo.b0 + et;
                if (bc < tl.B) atomicMax(chmax + bc, cm[et]);
                cm[et] = 0u;  // the next item adds to it after the barrier that follows its scale rows
            }
        }
    }

    __syncthreads();
    if (*abort_flag) {
        if (threadIdx.x == 0) atomicOr(status, kFlagTimeout);
        sleep_ns(200000);  // let in-flight copies and MMAs land before releasing memory
    }
    // PAIR: neither CTA leaves (or frees tensor memory) while the other may
    // still copy into, commit to or arrive on its shared memory
    if constexpr (PAIR) cluster_barrier();
    tc_fence_after();
    if (warp == 2) {
        if constexpr (PAIR)
            asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols)
                         : "memory");
        else
            asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols)
                         : "memory");
    }
}

// Item selection for channel b (blockIdx.y; blockIdx.x slices its entries).
// With bound[b] = 2 delta + 2 eps_r (k_shift_rows), as for the dense BF16
// search, the FP32 argmax lies in an item whose largest |h| is
// >= hmax - bound[b].  max_items: flagged items per channel before the full
// FP32 search.
__global__ void __launch_bounds__(256) k_shift_flag(int Ntc, int n_tiles, int bpt, int max_items,
                                                    const float *tile_max, const float *blk_max, const float *bound,
                                                    const unsigned int *chmax, const int *__restrict__ blk_order,
                                                    int *chcount, int *fb_list, int *counters, int *items,
                                                    long long *stats) {
    const int b = blockIdx.y;
    asm volatile("griddepcontrol.wait;" ::: "memory");  // the rows kernel's bound, the GEMM's maxima
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    // the threshold rounded down: a superset of the items
    // (what earlier kernels write is read through pointers without
    // __restrict__: a load that the compiler may take for constant could move
    // before the wait)
    const float thr_f = __fsub_rd(__uint_as_float(chmax[b]), bound[b]);
    // scan the tile maxima; a tile at or above the threshold is narrowed to
    // its 32-template blocks at or above it (the items: j * n_blocks + block)
    const float *tm = tile_max + (size_t)b * Ntc * n_tiles;
    const int n_entries = Ntc * n_tiles;
    const int n_blocks = n_tiles * bpt;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n_entries; i += gridDim.x * blockDim.x) {
        if (!(tm[i] >= thr_f)) continue;
        const int j = i / n_tiles, tile = i - j * n_tiles;
        const float4 *bm4 =
            reinterpret_cast<const float4 *>(blk_max + ((size_t)b * Ntc + j) * n_blocks + (size_t)tile * bpt);
        float bm[8];  // bpt is 4 or 8
        *reinterpret_cast<float4 *>(bm) = bm4[0];
        *reinterpret_cast<float4 *>(bm + 4) = bpt > 4 ? bm4[1] : make_float4(-1.f, -1.f, -1.f, -1.f);
        int hits = 0;
#pragma unroll
        for (int k = 0; k < 8; ++k) hits += k < bpt && bm[k] >= thr_f;
        if (hits == 0) continue;
        const int pos = atomicAdd(chcount + b, hits);
        const int take = max(0, min(hits, max_items - pos));
        if (pos <= max_items && pos + hits > max_items) {
            // too many: the FP32 search scores this channel in full
            fb_list[atomicAdd(&counters[0], 1)] = b;
            atomicAdd((unsigned long long *)&stats[1], 1ull);
            atomicAdd((unsigned long long *)&stats[0], ~0ull);  // -1: not resolved by the items
        }
        if (take == 0) continue;
        int at = atomicAdd(&counters[1], take);
        const int end = at + take;
        atomicAdd((unsigned long long *)&stats[2], (unsigned long long)take);
#pragma unroll
        for (int k = 0; k < 8; ++k)
            if (k < bpt && bm[k] >= thr_f && at < end) {
                items[2 * at] = b;
                items[2 * at + 1] = j * n_blocks + blk_order[tile * bpt + k];  // the templates' own block
                ++at;
            }
    }
}

// FP32 rescore, one warp per flagged (lag, 32-template block) item.  Lane =
// template.  Per phase a, the P template rows the FP32 template search reads
// for this lag (contiguous, P x 128 bytes) arrive by a bulk copy into one of
// the warp's nb buffers (the copies of the next nb - 1 phases are in flight
// while this one is used); each lane runs the FP32 search's FMA chain over
// them in its order and scales the sum the same way.  Each warp owns its
// barriers, buffers and residual phases; warps never wait on one another.
// Bound by latency: the item, the copies (all at once where nb = Sa) and the
// chain of L dependent FMAs.
__global__ void __launch_bounds__(kRescanWarps * 32) k_shift_rescan(
    const float *__restrict__ tpl, const float *__restrict__ scale, int S, int Sa, int P, int rows, int NtcP,
    int Ntc, int T, int n_blocks, int Lp, int L, const float *R, const int2 *items, int64_t max_tasks, int nb,
    const int *counters, unsigned long long *keys, int *status,
    unsigned long long wait_ns) {
    extern __shared__ __align__(128) float sm[];  // per warp: the residual [Lp], then nb x [P][32] rows
    __shared__ __align__(8) uint64_t bar[kRescanWarps][kRescanBufs];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const size_t buf_floats = (size_t)P * 32, warp_floats = (size_t)Lp + nb * buf_floats;
    float *rres = sm + warp * warp_floats;
    float *buf0 = rres + Lp;
    const uint32_t bytes = (uint32_t)P * 128u;
    const int nw = (int)(blockDim.x >> 5);
    if (lane < nb) mbar_init(&bar[warp][lane], 1);
    fence_mbar_init();
    __syncwarp();
    // tasks go to the first warp of every block before the second (one task
    // per SM while there are fewer tasks than SMs)
    const int64_t stride = (int64_t)gridDim.x * nw;
    int64_t task = (int64_t)warp * gridDim.x + blockIdx.x;
    asm volatile("griddepcontrol.wait;" ::: "memory");  // the flagged items
    // the first item is read beside the number of items, which says whether it
    // is one (neither may move before the wait: volatile, and no __restrict__)
    const volatile int2 *item_v = items;
    int2 item = make_int2(0, 0);
    if (task < max_tasks) item = make_int2(item_v[task].x, item_v[task].y);
    const int n_tasks = *(const volatile int *)&counters[1];  // at most kMaxItems per channel
    // the fallback search behind this kernel may launch now: it reads
    // nothing of ours before its wait for our completion
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    uint32_t par = 0u;  // bit i: the parity buffer i's next copy completes
    int cur_b = -1;
    for (bool first = true; task < n_tasks; task += stride, first = false) {
        if (!first) item = items[task];
        const int b = item.x;
        const int j = item.y / n_blocks, tb = item.y % n_blocks;
        if (tb * 32 >= T) continue;  // past the last template
        const float *src = tpl + ((size_t)tb * Sa * rows + (size_t)(NtcP - 1 - j)) * 32;
        auto copy = [&](int a, uint32_t more) {  // lane 0: phase a's rows into buffer a % nb
            uint64_t *br = &bar[warp][a % nb];
            mbar_expect_tx(br, bytes + more);
            bulk_g2s(buf0 + (size_t)(a % nb) * buf_floats, src + (size_t)a * rows * 32, bytes, br);
        };
        __syncwarp();
        if (lane == 0) {  // a new channel's residual with phase 0's rows
            const bool new_b = b != cur_b;
            copy(0, new_b ? (uint32_t)Lp * 4u : 0u);
            if (new_b) bulk_g2s(rres, R + (size_t)b * Lp, (uint32_t)Lp * 4u, &bar[warp][0]);
            for (int a = 1; a < nb && a < Sa; ++a) copy(a, 0u);
        }
        cur_b = b;
        // the scale is needed last: on its way meanwhile
        const float sc = scale[((size_t)tb * NtcP + j) * 32 + lane];
        float acc = 0.0f;
        for (int a = 0, cb = 0; a < Sa; ++a) {
            const int ok = mbar_wait(&bar[warp][cb], par >> cb & 1u, wait_ns) ? 1 : 0;
            if (!__all_sync(0xffffffffu, ok)) {
                if (lane == 0) {
                    atomicOr(status, kFlagTimeout);
                    // bounded: let the copies in flight land before the warp leaves
                    for (int f = a; f < Sa && f < a + nb; ++f) mbar_drain(&bar[warp][f % nb], par >> (f % nb) & 1u);
                }
                return;
            }
            par ^= 1u << cb;
            // sample n = a + S p of the window (0 past it, as in the FP32 search's phases)
            const float *bp = buf0 + (size_t)cb * buf_floats + lane;
#pragma unroll 8
            for (int p = 0; p < P; ++p) {
                const int n = a + S * p;
                acc = fmaf(n < L ? rres[n] : 0.0f, bp[p * 32], acc);
            }
            __syncwarp();
            if (a + nb < Sa && lane == 0) copy(a + nb, 0u);  // into the buffer just used
            if (++cb == nb) cb = 0;
        }
        const int t = tb * 32 + lane;
        unsigned long long key = 0ull;
        if (t < T) {
            const float sv = acc * sc;
            const float x = fabsf(sv);
            if (x == x) key = pack_key(x, (uint32_t)j * (uint32_t)T + (uint32_t)t);
        }
        for (int off = 16; off > 0; off >>= 1) {
            const unsigned long long o = __shfl_xor_sync(0xffffffffu, key, off);
            key = o > key ? o : key;
        }
        if (lane == 0 && key) atomicMax(keys + b, key);
    }
}

// static shared memory of the kernels here (the GEMM's Smem is the largest)
constexpr int kStaticReserve = 8192;
static_assert(sizeof(Smem) + 256 <= kStaticReserve, "static shared memory above its reserve");
constexpr int kSmemBudget = 232448 - kStaticReserve - 1024;

// Dynamic shared memory of a rescore block.  It has none of the GEMM's tables
// beside it, so its limit does not follow theirs: one warp with two buffers
// takes exactly these bytes at time centres one sample apart and windows of
// 849 to 864 samples, and two samples apart and 1,665 to 1,696, the longest
// windows that the tensor-core search serves at those steps.
constexpr int kRescanSmem = 225280;
static_assert(kRescanSmem + (int)sizeof(uint64_t) * kRescanWarps * kRescanBufs + 1024 <= 232448,
              "a rescore block's shared memory");

}  // namespace

struct ShiftTc {
    CUtensorMap mapB[2];    // box heights 128 and 256
    int nkc = 0, sm_count = 0, T_pad = 0;
    int pair_clusters = 0;  // co-resident CTA pairs of the paired GEMM (0: not available)
    int few_channels = 0;   // most channels of a call whose rescore takes rescan[0]
    struct {
        int bufs = 0, warps = 0, blocks_per_sm = 0;
        size_t smem = 0;
    } rescan[2];  // few channels, many
};

cudaError_t shift_tc_prepare(ShiftTc **out, const ShiftPlan &sp, int sm_count) {
    *out = nullptr;
    if (!sp.tpl16 || sp.Kt < kBK || sp.Kt % kBK != 0) return cudaErrorNotSupported;
    ShiftTc *s = new (std::nothrow) ShiftTc();
    if (!s) return cudaErrorMemoryAllocation;
    s->nkc = sp.Kt / kBK;
    s->T_pad = sp.T_pad;
    s->sm_count = sm_count;
    const uint64_t rows = (uint64_t)(sp.T_pad / kBlockRows) * s->nkc * kBlockRows;
    if (rows >= ((uint64_t)1 << 31) || !make_map(&s->mapB[0], sp.tpl16, (uint64_t)kBK, rows, 128) ||
        !make_map(&s->mapB[1], sp.tpl16, (uint64_t)kBK, rows, 256)) {
        delete s;
        return cudaErrorNotSupported;
    }
    const void *gemms[3] = {(const void *)k_shift_gemm<128, false>, (const void *)k_shift_gemm<256, false>,
                            (const void *)k_shift_gemm<256, true>};
    const int stage_bytes[3] = {ShiftTile<128>::kStageBytes, ShiftTile<256>::kStageBytes,
                                ShiftTile<256, true>::kStageBytes};
    cudaError_t e = cudaSuccess;
    for (int i = 0; i < 3 && e == cudaSuccess; ++i) e = allow_max_smem(gemms[i], 1024 + 2 * (size_t)stage_bytes[i]);
    if (e == cudaSuccess) e = allow_max_smem((const void *)k_shift_rows, 0);
    if (e == cudaSuccess) {
        // how many CTA pairs fit at once with the largest launch's shared memory
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = 2;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.gridDim = dim3(2 * (unsigned)sm_count);
        cfg.blockDim = dim3(kMaxThreads);
        cfg.dynamicSmemBytes = 1024 + (size_t)kSmemBudget;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int clusters = 0;
        if (cudaOccupancyMaxActiveClusters(&clusters, k_shift_gemm<256, true>, &cfg) != cudaSuccess) {
            cudaGetLastError();
            clusters = 0;
        }
        s->pair_clusters = clusters;
    }
    // rescore: per warp the residual and its P-row buffers; as many warps per
    // block (up to kRescanWarps) as fit
    const size_t buf = (size_t)sp.P * 128, res = sizeof(float) * (size_t)sp.Lp;
    size_t most = 0;
    for (int i = 0; i < 2; ++i) {
        int nb = 2;
        while (i == 0 && nb < sp.Sa && nb < kRescanBufs && res + (nb + 1) * buf <= (size_t)kRescanFewBytes) ++nb;
        if (i == 0) s->few_channels = nb < sp.Sa ? kRescanFewPhased : kRescanFewChannels;
        const size_t per_warp = res + nb * buf;
        int rw = kRescanWarps;
        while (rw > 1 && rw * per_warp > (size_t)kRescanSmem) --rw;
        s->rescan[i].bufs = nb;
        s->rescan[i].warps = rw;
        s->rescan[i].smem = rw * per_warp;
        most = s->rescan[i].smem > most ? s->rescan[i].smem : most;
        if (e == cudaSuccess && s->rescan[i].smem > (size_t)kRescanSmem) e = cudaErrorNotSupported;
    }
    if (e == cudaSuccess) e = allow_max_smem((const void *)k_shift_rescan, most);
    for (int i = 0; i < 2 && e == cudaSuccess; ++i) {
        int per_sm = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_shift_rescan, s->rescan[i].warps * 32,
                                                          s->rescan[i].smem);
        s->rescan[i].blocks_per_sm = per_sm < 1 ? 1 : per_sm;
    }
    if (e != cudaSuccess) {
        delete s;
        return e;
    }
    *out = s;
    return cudaSuccess;
}

void shift_tc_free(ShiftTc *s) { delete s; }

void shift_tc_scratch_free(ShiftTcScratch &x) {
    if (x.tile_max) cudaFree(x.tile_max);
    if (x.blk_max) cudaFree(x.blk_max);
    if (x.items) cudaFree(x.items);
    if (x.X) cudaFree(x.X);
    if (x.bound) cudaFree(x.bound);
    if (x.chmax) cudaFree(x.chmax);
    if (x.chcount) cudaFree(x.chcount);
    x = ShiftTcScratch();
}

// Row tiling for B channels: Bg channels x Jt time centres per 128-row tile,
// Jt as small as B allows (fewer lag chunks per tile), at most the time
// centres (rounded up to a power of two).  Up to 16 channels past whole
// blocks of 32 (up to 8 past one block of 16) take tiles of 8 or 16 channels x
// 16 or 8 time centres instead of one more block that is mostly padding,
// unless the time centres lie so far apart that such a tile's windows see over
// a quarter more lags.  Row build + GEMM in us per order with a padded block
// and with such tiles, EEG-like grid: 17 channels 41.0 and 36.7, 33 67.5 and
// 49.2, 48 68.3 and 57.5, 66 97 and 80; EMG-like, 2,048 samples: 90 and 78,
// 160 and 116, 167 and 141, 237 and 197; the uneven EMG-like batch (66, 60, 73
// and 57 channels) 25.1 and 21.2 ms.
static RowTiling make_tiling(const ShiftPlan &sp, int B) {
    RowTiling t;
    int bg = 1;
    while (bg < B && bg < 32) bg <<= 1;
    int ntc2 = 1;
    while (ntc2 < sp.Ntc) ntc2 <<= 1;
    t.Jt = kBM / bg < ntc2 ? kBM / bg : ntc2;
    t.Bg = kBM / t.Jt;
    t.B = B;
    t.Ntc = sp.Ntc;
    t.n_cb = (B + t.Bg - 1) / t.Bg;
    t.B_main = t.n_cb * t.Bg;
    t.Jt2 = t.Bg2 = 0;
    const int block = B > 32 ? 32 : 16, rest = B % block;
    if (B > 16 && t.Bg == 32 && rest > 0 && rest <= block / 2) {
        const int bg2 = rest <= 8 ? 8 : 16, jt2 = kBM / bg2;
        if (jt2 <= ntc2 && 4 * (int64_t)(jt2 - 1) * sp.S <= sp.L) {
            t.Bg = block;
            t.Jt = kBM / block;
            t.n_cb = B / block;
            t.B_main = t.n_cb * block;
            t.Bg2 = bg2;
            t.Jt2 = jt2;
        }
    }
    t.m_main = ((sp.Ntc + t.Jt - 1) / t.Jt) * t.n_cb;
    t.m_tiles = t.m_main + (t.Jt2 ? (sp.Ntc + t.Jt2 - 1) / t.Jt2 : 0);
    t.S = sp.S;
    t.L = sp.L;
    t.span0 = -sp.m_lo - sp.tc0;
    return t;
}

// Buffers for B channels (kept when large enough).
cudaError_t shift_tc_reserve(const ShiftTc *s, const ShiftPlan &sp, int B, ShiftTcScratch &x, cudaStream_t st) {
    (void)s;
    if (B <= x.B_cap) return cudaSuccess;
    shift_tc_scratch_free(x);
    const int64_t rows = (int64_t)B * sp.Ntc;
    int64_t rows_alloc = 0;  // the largest row-tile count of any B' <= B
    for (int b2 = 1; b2 <= B; ++b2) {
        const int64_t r2 = (int64_t)make_tiling(sp, b2).m_tiles * kBM;
        rows_alloc = r2 > rows_alloc ? r2 : rows_alloc;
    }
    if (rows_alloc > (1ll << 30)) return cudaErrorInvalidValue;
    cudaError_t e = dev_alloc((void **)&x.tile_max, sizeof(float) * (size_t)rows * (sp.T_pad / 128));
    if (e == cudaSuccess) e = dev_alloc((void **)&x.blk_max, sizeof(float) * (size_t)rows * (sp.T_pad / 32));
    if (e == cudaSuccess) e = dev_alloc((void **)&x.items, sizeof(int) * 2 * (size_t)B * kMaxItems);
    if (e == cudaSuccess) e = dev_alloc((void **)&x.X, sizeof(__nv_bfloat16) * (size_t)rows_alloc * sp.Kt);
    if (e == cudaSuccess) e = cudaMemsetAsync(x.X, 0, sizeof(__nv_bfloat16) * (size_t)rows_alloc * sp.Kt, st);
    if (e == cudaSuccess) e = dev_alloc((void **)&x.bound, sizeof(float) * (size_t)B);
    if (e == cudaSuccess) e = dev_alloc((void **)&x.chmax, sizeof(unsigned int) * (size_t)B);
    if (e == cudaSuccess) e = dev_alloc((void **)&x.chcount, sizeof(int) * (size_t)B);
    if (e != cudaSuccess) {
        cudaGetLastError();
        shift_tc_scratch_free(x);
        return cudaErrorMemoryAllocation;
    }
    x.B_cap = B;
    x.rows_alloc = (int)rows_alloc;
    return cudaSuccess;
}

// GEMM form of a B-channel launch: the template tile width (256 unless that
// leaves SMs idle or leaves room for fewer than two stages beside the tile's
// scale rows) and whether CTA pairs share each MMA (256-wide tiles, at least
// two row tiles, a work unit for every pair that fits, pairs allowed).  Two
// epilogue groups (*threads) where a second set of scale rows costs no stage
// below four.
static int shift_tc_bn(const ShiftTc *s, const ShiftPlan &sp, const RowTiling &tl, bool pairs_allowed, int *stages,
                       size_t *smem, bool *pair, int *threads) {
    auto smem_for = [&](int bn, int stage_bytes, int *stg_out) {
        const size_t sc = (size_t)(tl.Jt > tl.Jt2 ? tl.Jt : tl.Jt2) * (bn + 4) * sizeof(float);
        int groups = 2;
        int stg = (int)((kSmemBudget - 2 * (int64_t)sc) / stage_bytes);
        if (stg < 4) {
            groups = 1;
            stg = (int)((kSmemBudget - (int64_t)sc) / stage_bytes);
        }
        stg = stg > kMaxStages ? kMaxStages : stg;
        *stg_out = stg;
        *threads = 128 + 128 * groups;
        return 1024 + (size_t)stg * stage_bytes + groups * sc;
    };
    *pair = false;
    int st256 = 0;
    smem_for(256, ShiftTile<256>::kStageBytes, &st256);
    if ((int64_t)tl.m_tiles * (sp.T_pad / 256) >= s->sm_count && st256 >= 2) {
        int stp = 0;
        smem_for(256, ShiftTile<256, true>::kStageBytes, &stp);
        const int64_t units = (int64_t)((tl.m_tiles + 1) / 2) * (sp.T_pad / 256);
        if (pairs_allowed && s->pair_clusters > 0 && tl.m_tiles >= 2 && units >= s->pair_clusters && stp >= 2) {
            // the whole budget: every operand read of a stage's MMAs stays
            // inside the allocation even at the last stage
            static_assert((kMaxStages - 1) * ShiftTile<256, true>::kStageBytes + 48 * 1024 <= kSmemBudget,
                          "paired stages beyond the shared-memory budget");
            *pair = true;
            *stages = stp;
            *smem = 1024 + (size_t)kSmemBudget;
            return 256;
        }
        *smem = smem_for(256, ShiftTile<256>::kStageBytes, stages);
        return 256;
    }
    *smem = smem_for(128, ShiftTile<128>::kStageBytes, stages);
    return 128;
}

bool shift_tc_uses_pairs(const ShiftTc *s, const ShiftPlan &sp, int B, bool pairs_allowed) {
    if (!s || B < 1) return false;
    int stages = 0, threads = 0;
    size_t smem = 0;
    bool pair = false;
    shift_tc_bn(s, sp, make_tiling(sp, B), pairs_allowed, &stages, &smem, &pair, &threads);
    return pair;
}

cudaError_t launch_shift_tc_gemm(const ShiftTc *s, const ShiftTcScratch &x, const ShiftPlan &sp, const float *R,
                                 int Lp, int L, int B, int err_terms, long long *stats, int *status, cudaStream_t st,
                                 bool pdl, unsigned long long wait_ns, bool pairs_allowed) {
    if (!s || B < 1 || B > x.B_cap) return cudaErrorInvalidValue;
    const RowTiling tl = make_tiling(sp, B);
    // rows per block: up to 16, fewer when that leaves SMs idle (at least 4);
    // lag segments keep the 8 staged copies within 64 KB of shared memory
    int RJ = (int)(((int64_t)B * sp.Ntc + 2 * s->sm_count - 1) / (2 * s->sm_count));
    RJ = RJ < 4 ? 4 : (RJ > 16 ? 16 : RJ);
    constexpr int kRowsSmemSamples = 65536 / 18;  // samples per copy in 64 KB of 8 BF16 copies + the plain one
    while (RJ > 1 && sp.S * (RJ - 1) + 8 + 64 > kRowsSmemSamples) --RJ;
    int KSEG = sp.Kt;
    if (sp.S * (RJ - 1) + 8 + KSEG > kRowsSmemSamples) KSEG = (kRowsSmemSamples - 8 - sp.S * (RJ - 1)) / 64 * 64;
    if (KSEG < 64) return cudaErrorInvalidValue;
    const int n_seg = (sp.Kt + KSEG - 1) / KSEG;
    const int span_pad = (sp.S * (RJ - 1) + KSEG + 7) & ~7;
    const size_t rows_smem = ((size_t)9 * span_pad + 8) * sizeof(__nv_bfloat16);
    const int64_t gx = (int64_t)((sp.Ntc + RJ - 1) / RJ) * n_seg;
    if (gx >= ((int64_t)1 << 31) || B > 65535) return cudaErrorInvalidValue;
    cudaError_t e = launch_kernel(k_shift_rows, dim3((unsigned)gx, B), dim3(256), rows_smem, st, pdl, tl, R, Lp,
                                  sp.tc0, sp.m_lo, sp.Kt, RJ, KSEG, n_seg, span_pad, err_terms,
                                  (const unsigned int *)sp.eps_bits, x.X, x.bound, x.chmax, x.chcount, stats);
    if (e != cudaSuccess) return e;
    const int m_tiles = tl.m_tiles;
    CUtensorMap mapA;
    if (!make_map(&mapA, x.X, (uint64_t)sp.Kt, (uint64_t)m_tiles * kBM, kBM)) return cudaErrorInvalidValue;
    int stages = 0, threads = 0;
    size_t smem = 0;
    bool pair = false;
    const int bn = shift_tc_bn(s, sp, tl, pairs_allowed, &stages, &smem, &pair, &threads);
    const int n_tiles = sp.T_pad / bn;
    if (stages < 2) return cudaErrorInvalidValue;
    if (pair) {
        // clusters of 2: each CTA loads 128-template halves (box height 128)
        const int64_t units = (int64_t)((m_tiles + 1) / 2) * n_tiles;
        const int pairs = (int)(units < s->pair_clusters ? units : s->pair_clusters);
        return launch_kernel_cluster(k_shift_gemm<256, true>, dim3(2 * pairs), dim3(threads), smem, st, true, 2, mapA,
                                     s->mapB[0], tl, n_tiles, s->nkc, stages, sp.T_pad, (const short2 *)sp.span,
                                     (const float *)sp.scaleT, x.tile_max, x.blk_max, x.chmax, status, wait_ns);
    }
    const int i = bn == 256 ? 1 : 0;
    const int64_t items = (int64_t)m_tiles * n_tiles;
    const int grid = (int)(items < s->sm_count ? items : s->sm_count);
    // a programmatic dependent of the shifted-row build (set-up overlaps it)
    return launch_kernel(bn == 256 ? k_shift_gemm<256, false> : k_shift_gemm<128, false>, dim3(grid), dim3(threads),
                         smem, st, true, mapA, s->mapB[i], tl, n_tiles, s->nkc, stages, sp.T_pad,
                         (const short2 *)sp.span, (const float *)sp.scaleT, x.tile_max, x.blk_max, x.chmax, status,
                         wait_ns);
}

// Flags the items of every channel (first step of either resolve).
static cudaError_t launch_flag(const ShiftTc *s, const ShiftTcScratch &x, const ShiftPlan &sp, int B, int max_items,
                               int *fb_list, int *counters, long long *stats, cudaStream_t st, bool pdl) {
    const RowTiling tl = make_tiling(sp, B);
    int stages = 0, threads = 0;
    size_t smem = 0;
    bool pair = false;
    const int bn = shift_tc_bn(s, sp, tl, false, &stages, &smem, &pair, &threads);  // the GEMM's tile width
    const int n_tiles = sp.T_pad / bn;
    const int entries = sp.Ntc * n_tiles;
    int slices = (entries + 255) / 256;
    const int max_slices = (4 * s->sm_count + B - 1) / B;
    if (slices > max_slices) slices = max_slices;
    return launch_kernel(k_shift_flag, dim3(slices, B), dim3(256), 0, st, pdl, sp.Ntc, n_tiles, bn / 32, max_items,
                         (const float *)x.tile_max, (const float *)x.blk_max, (const float *)x.bound,
                         (const unsigned int *)x.chmax, (const int *)sp.blk_order, x.chcount, fb_list, counters,
                         x.items, stats);
}

cudaError_t launch_shift_tc_resolve(const ShiftTc *s, const ShiftTcScratch &x, const ShiftPlan &sp, const float *R,
                                    int Lp, int L, int B, unsigned long long *keys, int *fb_list, int *counters,
                                    long long *stats, int *status, cudaStream_t st, bool pdl,
                                    unsigned long long wait_ns) {
    if (!s || B < 1 || B > x.B_cap) return cudaErrorInvalidValue;
    cudaError_t e = launch_flag(s, x, sp, B, kMaxItems, fb_list, counters, stats, st, pdl);
    if (e != cudaSuccess) return e;
    const auto &rc = s->rescan[B <= s->few_channels ? 0 : 1];
    e = launch_kernel(k_shift_rescan, dim3(s->sm_count * rc.blocks_per_sm), dim3(rc.warps * 32), rc.smem, st, true,
                      (const float *)sp.tpl, (const float *)sp.scale, sp.S, sp.Sa, sp.P, sp.rows, sp.NtcP, sp.Ntc,
                      sp.T, sp.T_pad / 32, Lp, L, R, reinterpret_cast<const int2 *>(x.items),
                      (int64_t)x.B_cap * kMaxItems, rc.bufs, (const int *)counters, keys, status, wait_ns);
    if (e != cudaSuccess) return e;
    // channels with more than kMaxItems flagged items: the FP32 template
    // search over the queue, launched early (its CTAs become resident while
    // the rescore runs and read the queue after it; an empty queue leaves
    // them idle)
    return launch_shift_search(sp, R, Lp, L, B, keys, nullptr, status, true, st, fb_list, &counters[0], wait_ns);
}

cudaError_t launch_shift_tc_resolve_rows(const ShiftTc *s, const ShiftTcScratch &x, const ShiftPlan &sp,
                                         const float *D32, int64_t K, const float *R, int Lp, int L, int B,
                                         unsigned long long *keys, int *fb_list, int *counters, long long *stats,
                                         int *status, int gemv_grid, cudaStream_t st, bool pdl,
                                         unsigned long long wait_ns) {
    if (!s || B < 1 || B > x.B_cap) return cudaErrorInvalidValue;
    cudaError_t e = launch_flag(s, x, sp, B, kMaxRowItems, fb_list, counters, stats, st, pdl);
    if (e == cudaSuccess)
        e = launch_rows_rescan(D32, K, Lp, R, x.items, counters, keys, sp.T, sp.T_pad / 32, s->sm_count, st);
    if (e != cudaSuccess) return e;
    return launch_gemv_argmax(D32, K, Lp, R, B, fb_list, &counters[0], keys, status, gemv_grid, st, wait_ns, true);
}

}  // namespace act
