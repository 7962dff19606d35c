// LEM-inspired hierarchical coarse-to-fine search (Sec. VII-A, Fig. 7), with
// no stored dictionary: per channel and order,
//   1. a Latin hypercube sample of n_coarse parameter vectors over the grid's
//      box (strata ranked by SplitMix64 keys, uniform offsets inside them);
//   2. every candidate atom generated on the fly and projected onto the
//      residual; the top_k by |score| kept (lowest candidate index on ties,
//      duplicate parameter vectors skipped);
//   3. per refinement level, the local neighbourhood dictionary of each kept
//      candidate (offsets -R..R steps of that level per axis, clamped to the
//      box), all candidates pooled, projected and reranked to a new top_k;
//      (2 and 3 as two kernels a level: k_lem_screen projects every candidate
//      in plain FP32 with an error bound, k_lem_pick projects again, in
//      float-float, those that the bound leaves among the top_k, and keeps
//      the top_k by that score: the selection is the float-float score's)
//   4. the best candidate then starts the BFGS refinement (act_refine.cu).
// The random draws come from SplitMix64 (Steele, Lea and Flood, 2014): draw
// n of a stream seeded s is mix(s + (n + 1) 0x9E3779B97F4A7C15), with n
// packing (channel, order, axis, kind, sample).
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "act_device.cuh"
#include "act_ff.cuh"
#include "act_internal.cuh"

namespace act {

namespace {

constexpr int kLemThreads = 256;

__device__ __forceinline__ uint64_t splitmix64_at(uint64_t seed, uint64_t n) {
    uint64_t z = seed + (n + 1ull) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

__device__ __forceinline__ uint64_t lem_counter(int channel, int order, int axis, int kind, int i) {
    return (((((((uint64_t)channel << 12) | (uint64_t)order) << 2 | (uint64_t)axis) << 1) | (uint64_t)kind) << 20) |
           (uint64_t)i;
}

// 1. Latin hypercube: one block per (channel, axis).  The stratum of sample i
// is the rank of its key (all keys of a call differ: SplitMix64's mix is a
// bijection).  The keys are uniform, so the rank comes from 2^log2b >= n / 2
// buckets of the leading bits: count, scan, gather, and compare within the
// bucket (a key or two each).  Five barriers; a bitonic sort of 2,048 keys
// took 66 steps (69 us against 15 per order at 64 channels).
constexpr int kLhsThreads = 512;

__global__ void __launch_bounds__(kLhsThreads) k_lem_lhs(int n, int log2b, LemBox box, uint64_t seed, int order,
                                                        int cap, double *cand, int *ncand) {
    // The samples do not depend on the residual: this kernel runs beside the
    // update of the order before it.  Nothing else reads or writes cand and
    // ncand by then (the update's own predecessors have completed before it
    // lets this kernel launch), and the wait at the end makes the screening
    // behind this kernel wait for the update too.
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    extern __shared__ uint8_t sm_raw[];
    __shared__ uint32_t part[kLhsThreads / 32];
    const int nb = 1 << log2b;
    uint64_t *key = reinterpret_cast<uint64_t *>(sm_raw);         // [n] gathered by bucket
    uint32_t *start = reinterpret_cast<uint32_t *>(key + n);      // [nb] first position of each bucket
    uint32_t *fill = start + nb;                                  // [nb] keys counted, then gathered
    const int b = blockIdx.x, a = blockIdx.y;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double *out = cand + (size_t)b * cap * 4;
    auto bucket = [&](uint64_t k) { return log2b ? (uint32_t)(k >> (64 - log2b)) : 0u; };
    for (int i = threadIdx.x; i < nb; i += blockDim.x) fill[i] = 0u;
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += blockDim.x)
        atomicAdd(&fill[bucket(splitmix64_at(seed, lem_counter(b, order, a, 0, i)))], 1u);
    __syncthreads();
    // exclusive scan: each thread its run of buckets, then the warps, then the block
    const int per = (nb + (int)blockDim.x - 1) / (int)blockDim.x;
    const int lo = min(nb, (int)threadIdx.x * per), hi = min(nb, lo + per);
    uint32_t sum = 0u;
    for (int i = lo; i < hi; ++i) sum += fill[i];
    uint32_t incl = sum;
    for (int off = 1; off < 32; off <<= 1) {
        const uint32_t v = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += v;
    }
    if (lane == 31) part[warp] = incl;
    __syncthreads();
    uint32_t at = incl - sum;
    for (int w = 0; w < warp; ++w) at += part[w];
    for (int i = lo; i < hi; ++i) {
        const uint32_t c = fill[i];
        start[i] = at;
        fill[i] = 0u;
        at += c;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const uint64_t k = splitmix64_at(seed, lem_counter(b, order, a, 0, i));
        const uint32_t q = bucket(k);
        key[start[q] + atomicAdd(&fill[q], 1u)] = k;
    }
    __syncthreads();
    // For n a power of two the quotient (p + u) / n is the exact product with
    // 2^-k: the same correctly rounded value without an FP64 division
    const bool pow2 = (n & (n - 1)) == 0;
    const double inv_n = pow2 ? __longlong_as_double((long long)(1023 - (31 - __clz(n))) << 52) : 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const uint64_t k = splitmix64_at(seed, lem_counter(b, order, a, 0, i));
        const uint32_t q = bucket(k), s0 = start[q], s1 = s0 + fill[q];
        uint32_t p = s0;  // the rank
        for (uint32_t e = s0; e < s1; ++e) p += key[e] < k ? 1u : 0u;
        const uint64_t h = splitmix64_at(seed, lem_counter(b, order, a, 1, i));
        const double u = (double)(h >> 11) * 0x1.0p-53;
        const double v = __dadd_rn((double)p, u);
        const double t = pow2 ? __dmul_rn(v, inv_n) : __ddiv_rn(v, (double)n);
        out[4 * i + a] = __dadd_rn(box.lo[a], __dmul_rn(t, __dadd_rn(box.hi[a], -box.lo[a])));
    }
    if (threadIdx.x == 0 && a == 0) ncand[b] = n;
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// The candidate that offset o (0 .. per - 1, c fastest) of the neighbourhood
// of kept parameters th names, clamped to the box.
__device__ __forceinline__ void lem_neighbour(const double *__restrict__ th, int o, const LemBox &box,
                                              const LemLevel &lev, double *p) {
#pragma unroll
    for (int a = 3; a >= 0; --a) {
        const int w = 2 * lev.radius[a] + 1;
        const double v = __dadd_rn(th[a], __dmul_rn((double)(o % w - lev.radius[a]), lev.step[a]));
        o /= w;
        p[a] = v < box.lo[a] ? box.lo[a] : (v > box.hi[a] ? box.hi[a] : v);
    }
}

// 2. Screening: h = |<r, u>| / |u| of every candidate in plain FP32, and a
// bound c with |h - |s|| <= c |r| for the float-float score s of
// lem_score_warp.  Per sample:
//  * the phase in cycles is a 32-bit fixed-point recurrence (wrapping is the
//    reduction mod 1): phi(n) = A + B n + C n^2 with A, B, C rounded to
//    2^-64, a lane's first phase and differences from those, then two
//    integer adds a sample; its leading 23 bits become a float by one shift;
//  * cos and exp by the hardware approximations (the sign that the half-cycle
//    shift of the float form costs is lost in |h|);
//  * samples beyond kScreenX durations from the centre are left out.
// The bound, with x = (n - tc) / (fs dt), e the envelope, x0 = |x| of the
// window's nearest sample, K <= 64 samples a lane, relative to |e|_2:
//  * phase: 2 pi (2^-32 (1 + K + K^2 / 2) + 2^-24) radians; cos.approx 2^-20.9
//    absolute on [-pi, pi]; 2 pi y and its scaling inside cos 4 2^-24 pi;
//  * envelope: forming x rounds 2^-24 of at most 2 kScreenX four times, its
//    step (expf 2 ulp, three products) is off by 5.4e-7 of itself, the
//    exponents round to 2.2e-7 of themselves over both sides, ex2.approx and
//    expf 2 ulp each: |x| 1.7e-6 + x^2 8e-7 + 5e-7, and under the weights
//    e^2 of the samples x counts as at most x0 + 1.5;
//  * the samples left out: below 2e-6 |e| while x0 <= 2;
//  * the FP32 sums of either side: (K + 40) 2^-24 |u| for <r, u> and for |u|.
// The first three act as twice a perturbation of u, relative to |u|: they
// count 2 |e| / |u|, where |e|^2 <= sqrt(pi) / dx + 1 (the integral of
// exp(-x^2) plus its largest term, dx = the step of x).  The whole is
// doubled; measured over EEG-, EMG- and radar-like, sub-sample, long and
// off-window candidates the largest error was 0.014 of the bound.
// Where x0 > 2, or the sums are so small that squares vanish, or the phase
// so large that FP64 does not hold it, c is infinite: k_lem_pick then always
// projects the candidate again.
// Bound by instruction issue (three slots of four busy; the special-function
// pipe is a quarter used) beside the FP64 set-up of a block's candidates: 44
// us for 64 channels x 2,048 candidates x 512 samples, where the float-float
// projection of all takes 230 us (118 instructions a sample).  The phase's
// products are formed once per candidate, a lane adds its own few (every lane
// forming them: 1 % per decomposition).  Slower or no faster: the cosine as
// a polynomial on the FMA pipe (6 %), two samples to a packed instruction (48
// registers: fewer warps), 32 candidates a block, 32 registers a thread.
constexpr float kScreenX = 5.8f;
constexpr int kScreenCands = 64;
constexpr float kScreenWide = 2.0f;

struct ScreenConst {
    uint64_t P, P1, C;    // phase of sample 32 row_lo + l: P + P1 l + C l^2, in 2^-64 cycles
    uint64_t D32;         // its difference over 32 samples, at l = 0
    float xs, dx;         // sqrt(log2(e) / 2) x of sample 32 row_lo, and its step per sample
    int row_lo, row_hi;   // rows of 32 samples projected
    float c_u, c_s;       // error bound: (c_u / |u| + c_s) |r|
};

__device__ __forceinline__ uint64_t cycles64(double v) {
    return (uint64_t)__double2ll_rn((v - rint(v)) * 0x1.0p64);  // saturates at half a cycle: 2^-64 off
}

__global__ void __launch_bounds__(kLemThreads) k_lem_screen(int cap, int level, LemBox box, LemLevel lev, int top_k,
                                                           const double *kept, const int *nkept, double *cand,
                                                           int *ncand, const float *R, int Lp, int L, double inv_fs,
                                                           float2 *screen) {
    // (no __restrict__ on what earlier kernels write: loads through it may
    // move ahead of the wait)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    extern __shared__ float r_sm[];  // the residual, zero up to a whole row
    __shared__ ScreenConst ks[kScreenCands];
    // every lane's <r, u> and |u|^2 of every candidate: added up by one
    // thread each at the end (a shuffle tree per sum cost as much as 8 samples)
    __shared__ float sums[2 * kScreenCands][33];
    const int b = blockIdx.y;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int i0 = blockIdx.x * kScreenCands;
    int n_cand, per = 1;
    if (level == 0) {
        n_cand = ncand[b];
    } else {
#pragma unroll
        for (int a = 0; a < 4; ++a) per *= 2 * lev.radius[a] + 1;
        n_cand = nkept[b] * per;
    }
    const int n_here = min(kScreenCands, n_cand - i0);
    if (n_here <= 0) return;  // the first block always has candidates: nkept >= 1 unless no score is a number
    if (threadIdx.x < n_here) {
        const int i = i0 + threadIdx.x;
        double *th = cand + ((size_t)b * cap + i) * 4;
        double p[4];
        if (level == 0) {
#pragma unroll
            for (int a = 0; a < 4; ++a) p[a] = th[a];
        } else {  // the candidates of this level, for k_lem_pick too
            lem_neighbour(kept + ((size_t)b * top_k + i / per) * 4, i % per, box, lev, p);
#pragma unroll
            for (int a = 0; a < 4; ++a) th[a] = p[a];
        }
        ScreenConst k;
        const double g = p[3] * inv_fs * inv_fs, f = p[1] * inv_fs, gt = g * p[0];
        const double alpha = (gt - f) * p[0], beta = f - 2.0 * gt;
        const uint64_t A = cycles64(alpha), B = cycles64(beta), C = cycles64(g);
        const float big = (float)(fabs(gt * p[0]) + fabs(f * p[0]) + fabs(beta) * L) + fabsf((float)g) * L * (float)L;
        // 1 / dt = exp(-logdt), the argument's rounding made good
        const float ah = (float)-p[2], al = (float)(-p[2] - (double)ah);
        const float dx = expf(ah) * (1.0f + al) * (float)inv_fs;  // x per sample
        const float nearest = fminf(fmaxf(rintf((float)p[0]), 0.0f), (float)(L - 1));
        const float x0 = fabsf((float)((double)nearest - p[0])) * dx;
        const float reach = kScreenX / dx;
        const float lo = (float)p[0] - reach, hi = (float)p[0] + reach;
        k.row_lo = lo > 0.0f ? (lo < (float)L ? (int)lo >> 5 : L) : 0;
        k.row_hi = hi < (float)L ? (hi >= 0.0f ? ((int)hi + 1 >> 5) + 1 : 0) : (L + 31) >> 5;
        k.row_hi = min(k.row_hi, (L + 31) >> 5);
        const uint64_t n0 = 32ull * (uint64_t)k.row_lo;
        k.P = A + (B + C * n0) * n0;
        k.P1 = B + 2ull * C * n0;
        k.C = C;
        k.D32 = 32ull * (B + C * (2ull * n0 + 32ull));
        constexpr float kScale = 0.84932180f;  // sqrt(log2(e) / 2)
        k.dx = dx * kScale;
        k.xs = (float)((double)(32 * k.row_lo) - p[0]) * k.dx;
        const float K = (float)(k.row_hi - k.row_lo), w = x0 + 1.5f;
        const float a_phase = 6.2831853f * (2.3283064e-10f * (1.0f + K + 0.5f * K * K) + 5.9604645e-8f);
        const float a_cos = a_phase + 5.1e-7f + 7.6e-7f;
        const float a_env = w * 1.7e-6f + w * w * 8e-7f + 5e-7f;
        k.c_u = 2.0f * 2.0f * (a_cos + a_env + 2e-6f) * sqrtf(1.7724539f / dx + 1.0f);
        k.c_s = 2.0f * 2.0f * (K + 40.0f) * 5.9604645e-8f;
        // not covered by the bound (comparisons written so that a NaN is not either)
        if (!(x0 <= kScreenWide && big <= 1e6f && dx >= 1e-20f && dx <= 1e6f)) k.c_u = __int_as_float(0x7f800000);
        ks[threadIdx.x] = k;
    }
    const int rows = (L + 31) >> 5;
    const float *r = R + (size_t)b * Lp;
    for (int n = threadIdx.x; n < rows * 32; n += blockDim.x) r_sm[n] = n < L ? r[n] : 0.0f;
    __syncthreads();
    constexpr int kWarps = kLemThreads / 32;
    const uint64_t lu = (uint64_t)lane;
    for (int q = warp; q < n_here; q += kWarps) {
        const ScreenConst k = ks[q];
        // phase of the lane's first sample and its differences over 32 and 32
        // samples (+ 256: the shift below rounds)
        uint32_t ph = (uint32_t)((k.P + lu * k.P1 + (lu * lu) * k.C) >> 32) + 256u;
        uint32_t d1 = (uint32_t)((k.D32 + (64ull * lu) * k.C) >> 32);
        const uint32_t d2 = (uint32_t)((2048ull * k.C) >> 32);
        const float x_lane = fmaf((float)lane, k.dx, k.xs), step = 32.0f * k.dx;
        float ru = 0.0f, uu = 0.0f;
        auto sample = [&](float x, float rv, bool in) {
            float e;
            asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(-x * x));
            e = in ? e : 0.0f;
            const float y = __uint_as_float(__funnelshift_r(ph, 0x7fu, 9));  // 1 + the phase
            const float u = e * __cosf(fmaf(6.2831853f, y, -9.4247780f));   // less half a cycle
            ph += d1;
            d1 += d2;
            ru = fmaf(rv, u, ru);
            uu = fmaf(u, u, uu);
        };
        const float *rp = r_sm + 32 * k.row_lo + lane;
        const int whole = min(k.row_hi, L >> 5) - k.row_lo;  // rows without an end in them
        int t = 0;
        for (; t + 4 <= whole; t += 4) {
            const float xb = fmaf((float)t, step, x_lane);
#pragma unroll
            for (int e = 0; e < 4; ++e) sample(fmaf((float)e, step, xb), rp[32 * (t + e)], true);
        }
        for (; t < k.row_hi - k.row_lo; ++t)
            sample(fmaf((float)t, step, x_lane), rp[32 * t], 32 * (k.row_lo + t) + lane < L);
        sums[2 * q][lane] = ru;
        sums[2 * q + 1][lane] = uu;
    }
    __syncthreads();
    if (threadIdx.x < 2 * kScreenCands) {
        float v = 0.0f;
        if (threadIdx.x < 2 * n_here)
            for (int l = 0; l < 32; ++l) v += sums[threadIdx.x][l];
        const float uu = __shfl_down_sync(0xffffffffu, v, 1);
        const int q = threadIdx.x >> 1;
        if (!(threadIdx.x & 1) && q < n_here) {
            const float inv = rsqrtf(uu);
            screen[(size_t)b * cap + i0 + q] = make_float2(
                fabsf(v) * inv, uu >= 1e-18f ? ks[q].c_u * inv * 1.001f + ks[q].c_s : __int_as_float(0x7f800000));
        }
    }
}

// The score s = <r, u> / |u| of one candidate by one warp, lane = sample
// stride 32.  A lane's samples n_k = lane + 32 k advance tau by D = 32 / fs,
// so the phase (c tau + fc) tau steps by d1_k = D (c (2 tau_k + D) + fc), and
// d1 by d2 = 2 c D^2: tau, the phase and d1 are carried by these recurrences
// in float-float (phase and d1 mod 1), from exact starting values at k = 0.
// The samples are FP32 from the same expressions as the dictionary
// generator's; products are summed in FP32 over 4 samples, then into
// float-float sums.
struct LemConst {
    ChirpFF k;
    ff D, d2;  // the lane stride in tau and the second difference of the phase (mod 1)
};

__device__ __forceinline__ LemConst lem_const(const double *__restrict__ th, double inv_fs) {
    const double D = 32.0 * inv_fs;
    double d2 = 2.0 * th[3] * D * D;
    d2 -= rint(d2);
    return {chirp_ff(th[0], inv_fs, th[1], th[3], exp(-th[2])), ff_from_double(D), ff_from_double(d2)};
}

__device__ __forceinline__ void lem_score_warp(const LemConst &kc, const float *__restrict__ r, int L, int lane,
                                               ff &ru, ff &uu) {
    const ChirpFF &k = kc.k;
    // k = 0: tau, the phase and its first difference, formed directly
    ff tau;
    ff ph = chirp_phase_pair(lane, k, &tau);
    const ff two_tau_d = ff_add({2.0f * tau.hi, 2.0f * tau.lo}, kc.D);
    ff d1 = ff_frac(ff_mul(ff_add(ff_mul(k.c, two_tau_d), k.fc), kc.D));
    ru = {0.0f, 0.0f};
    uu = {0.0f, 0.0f};
    for (int n0 = lane; n0 < L; n0 += 128) {
        float pr = 0.0f, pu = 0.0f;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int n = n0 + 32 * e;
            if (n < L) {
                const float x = chirp_x_ff(tau, k);
                const float u = expf(-0.5f * x * x) * cospif(2.0f * (ph.hi + ph.lo));
                pr = fmaf(r[n], u, pr);
                pu = fmaf(u, u, pu);
                tau = ff_add_sloppy(tau, kc.D);
                ph = ff_frac(ff_add_sloppy(ph, d1));
                d1 = ff_frac(ff_add_sloppy(d1, kc.d2));
            }
        }
        ru = ff_add_f(ru, pr);
        uu = ff_add_f(uu, pu);
    }
    ru = ff_warp_sum(ru);
    uu = ff_warp_sum(uu);
}

// 3. The top_k of one channel by float-float score, one block per channel.
// Compares run on bit patterns (integer pipes; FP64 compares are slow on
// this GPU): for finite non-negative values the patterns order as the
// values, NaN scores are skipped, and two parameters are equal when their
// patterns are, or both are zeros.
__device__ __forceinline__ bool same_value(unsigned long long a, unsigned long long b) {
    return a == b || ((a | b) << 1) == 0ull;
}

constexpr int kPickThreads = 512;
constexpr int kPickList = 1024;   // candidates projected again that the block holds in a list
constexpr int kPickBatch = 256;   // of these, whose constants are held at once
constexpr int kMaxTopK = 16;

struct PickShared {
    unsigned long long bv[2][kPickThreads / 32];  // by the parity of the choice
    int bi[2][kPickThreads / 32];
    int chosen[kMaxTopK];
    unsigned long long value[kMaxTopK];
    float sum[kPickThreads / 32];
    int count;
    int list[kPickList];
    LemConst consts[kPickBatch];
};

// The best (v, i) of the warp, by three reductions: largest v, then lowest i
// (i >= 0 names a candidate); the same for all lanes.
__device__ __forceinline__ void warp_best(unsigned long long &v, int &i) {
    const uint32_t hi = (uint32_t)(v >> 32), lo = (uint32_t)v;
    const uint32_t mh = __reduce_max_sync(0xffffffffu, i >= 0 ? hi : 0u);
    const uint32_t ml = __reduce_max_sync(0xffffffffu, i >= 0 && hi == mh ? lo : 0u);
    const uint32_t mi = __reduce_min_sync(0xffffffffu, i >= 0 && hi == mh && lo == ml ? (uint32_t)i : 0xffffffffu);
    v = ((unsigned long long)mh << 32) | ml;
    i = (int)mi;  // -1: no candidate
}

// Up to k candidates by value(i) (0: not a candidate), largest first, the
// lowest index among equals, a parameter vector already chosen skipped (equal
// parameters have equal values, so only those of equal value are compared).
// Each thread holds the best of its own entries e = tid, tid + threads, ...
// (index_of(e)) and looks for its next one only when that is chosen or
// repeats a choice: the first kHeld of them stay in registers (reading them
// again from L2 was most of the time).  One barrier per choice.  Returns how
// many were found, the same for all threads.
template <typename IndexOf, typename Value>
__device__ int pick_top(PickShared &sm, int k, int entries, const unsigned long long *__restrict__ cb, IndexOf index_of,
                        Value value) {
    constexpr int kHeld = 4;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned long long hv[kHeld];
#pragma unroll
    for (int h = 0; h < kHeld; ++h) {
        const int e = threadIdx.x + h * kPickThreads;
        hv[h] = e < entries ? value(index_of(e)) : 0ull;
    }
    unsigned long long mv = 0ull;
    int mi = -1;
    // the best of this thread's entries that come after (v, i) in the order
    auto next_after = [&](unsigned long long v, int i, bool first) {
        mv = 0ull;
        mi = -1;
        auto offer = [&](int c, unsigned long long x) {
            if (x == 0ull || (!first && (x > v || (x == v && c <= i)))) return;
            if (mi < 0 || x > mv || (x == mv && c < mi)) {
                mv = x;
                mi = c;
            }
        };
#pragma unroll
        for (int h = 0; h < kHeld; ++h)
            if (hv[h]) offer(index_of(threadIdx.x + h * kPickThreads), hv[h]);
        for (int e = threadIdx.x + kHeld * kPickThreads; e < entries; e += kPickThreads) {
            const int c = index_of(e);
            offer(c, value(c));
        }
    };
    auto repeats = [&](int i, int j) {
        if (i == j) return true;
        unsigned long long x[4], y[4];
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            x[a] = cb[4 * (size_t)i + a];
            y[a] = cb[4 * (size_t)j + a];
        }
        return same_value(x[0], y[0]) && same_value(x[1], y[1]) && same_value(x[2], y[2]) && same_value(x[3], y[3]);
    };
    next_after(0ull, 0, true);
    int m = 0;
    for (; m < k; ++m) {
        unsigned long long v = mv;
        int i = mi;
        warp_best(v, i);
        if (lane == 0) {
            sm.bv[m & 1][warp] = v;
            sm.bi[m & 1][warp] = i;
        }
        __syncthreads();
        // every warp finds the block's best for itself
        constexpr int kWarps = kPickThreads / 32;
        v = lane < kWarps ? sm.bv[m & 1][lane] : 0ull;
        i = lane < kWarps ? sm.bi[m & 1][lane] : -1;
        warp_best(v, i);
        if (i < 0) break;  // nothing left
        // read back below by this warp alone before the next barrier; all warps write the same
        if (lane == 0) {
            sm.chosen[m] = i;
            sm.value[m] = v;
        }
        __syncwarp();
        while (mi >= 0) {  // this thread's best that repeats no choice
            bool dup = false;
            for (int q = m; q >= 0 && sm.value[q] == mv && !dup; --q) dup = repeats(mi, sm.chosen[q]);
            if (!dup) break;
            next_after(mv, mi, false);
        }
    }
    __syncthreads();
    return m;
}

__global__ void __launch_bounds__(kPickThreads) k_lem_pick(int cap, int k, int level_candidates,
                                                          const double *cand, const int *ncand, int per, int *nkept,
                                                          const float2 *screen, const float *R, int Lp, int L,
                                                          double inv_fs, double *score, double *kept,
                                                          double *kept_score) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    constexpr unsigned long long kAbs = 0x7fffffffffffffffull, kInf = 0x7ff0000000000000ull;
    extern __shared__ __align__(16) uint8_t pick_raw[];
    PickShared &sm = *reinterpret_cast<PickShared *>(pick_raw);
    const int b = blockIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int n = level_candidates ? nkept[b] * per : ncand[b];
    const double *cd = cand + (size_t)b * cap * 4;
    const unsigned long long *cb = reinterpret_cast<const unsigned long long *>(cd);
    const float2 *sc = screen + (size_t)b * cap;
    double *ss = score + (size_t)b * cap;
    const float *r = R + (size_t)b * Lp;
    // |r| from above: an FP32 sum of at most 2048 squares is within 1.3e-4
    // relative of the exact one, and squares that underflow lose less than 1e-18
    float e = 0.0f;
    int nonzero = 0;
    for (int i = threadIdx.x; i < L; i += kPickThreads) {
        const float x = r[i];
        e = fmaf(x, x, e);
        nonzero |= x != 0.0f;
    }
    e = warp_sum(e);
    if (lane == 0) sm.sum[warp] = e;
    if (threadIdx.x == 0) sm.count = 0;
    const bool zero = !__syncthreads_or(nonzero);
    float tot = 0.0f;
    for (int w = 0; w < kPickThreads / 32; ++w) tot += sm.sum[w];
    const float rn = sqrtf(tot) * 1.001f + 1e-18f;

    int entries = n;
    bool listed = false;
    float thr = -__int_as_float(0x7f800000);
    // h + c |r|, rounded up; not below thr, or not a number: to be projected again
    auto in_reach = [&](int i) { return !(__fadd_ru(sc[i].x, __fmul_ru(sc[i].y, rn)) < thr); };
    if (!zero) {
        // the k-th largest lower bound h - c |r| over distinct parameters:
        // the top_k scores are at least that
        const int m = pick_top(
            sm, k, n, cb, [](int e2) { return e2; },
            [&](int i) {
                const float lo = __fadd_rd(sc[i].x, -__fmul_ru(sc[i].y, rn));
                return lo >= 0.0f ? (unsigned long long)__float_as_uint(lo) + 1ull : 0ull;
            });
        if (m == k) thr = __uint_as_float((unsigned)(sm.value[k - 1] - 1ull));
        __syncthreads();
        for (int i = threadIdx.x; i < n; i += kPickThreads)
            if (in_reach(i)) {
                const int at = atomicAdd(&sm.count, 1);
                if (at < kPickList) sm.list[at] = i;
            }
        __syncthreads();
        const int count = sm.count;
        listed = count <= kPickList;
        if (listed) entries = count;
        auto finish = [&](ff ru, ff uu) {
            const double en = ff_to_double(uu);
            return (en > 0.0 && isfinite(en)) ? ff_to_double(ru) / sqrt(en) : 0.0;
        };
        // the same steps for listed candidates and, past the list, for all in reach
        for (int e0 = 0; e0 < entries; e0 += kPickBatch) {
            const int here = min(kPickBatch, entries - e0);
            if (threadIdx.x < here) {
                const int i = listed ? sm.list[e0 + threadIdx.x] : e0 + threadIdx.x;
                if (listed || in_reach(i)) sm.consts[threadIdx.x] = lem_const(cd + 4 * (size_t)i, inv_fs);
            }
            __syncthreads();
            // lane q keeps the sums of the warp's q-th candidate: the FP64
            // finish runs once for all of them
            ff my_ru = {0.0f, 0.0f}, my_uu = {0.0f, 0.0f};
            int mine = -1, q = 0;
            for (int t = warp; t < here; t += kPickThreads / 32) {
                const int i = listed ? sm.list[e0 + t] : e0 + t;
                if (!listed && !in_reach(i)) continue;
                ff ru, uu;
                lem_score_warp(sm.consts[t], r, L, lane, ru, uu);
                if (lane == q) {
                    my_ru = ru;
                    my_uu = uu;
                    mine = i;
                }
                ++q;
            }
            if (mine >= 0) ss[mine] = finish(my_ru, my_uu);
            __syncthreads();
        }
    }
    // a zero residual scores 0 everywhere
    const int m = pick_top(
        sm, k, entries, cb, [&](int e2) { return listed ? sm.list[e2] : e2; },
        [&](int i) {
            if (zero) return 1ull;
            if (!listed && !in_reach(i)) return 0ull;
            const unsigned long long v = (unsigned long long)__double_as_longlong(ss[i]) & kAbs;
            return v > kInf ? 0ull : v + 1ull;
        });
    if (threadIdx.x < m) {
        const int i = sm.chosen[threadIdx.x];
        kept_score[(size_t)b * k + threadIdx.x] = zero ? 0.0 : ss[i];
#pragma unroll
        for (int a = 0; a < 4; ++a) kept[((size_t)b * k + threadIdx.x) * 4 + a] = cd[4 * (size_t)i + a];
    }
    if (threadIdx.x == 0) nkept[b] = m;
}

}  // namespace

cudaError_t launch_lem_select(const LemConfig &cfg, int B, int order, const float *R, int Lp, int L, double fs,
                              const LemBuffers &lb, cudaStream_t st, bool pdl) {
    int log2b = 0;
    while ((1 << log2b) < cfg.n_coarse && log2b < 13) ++log2b;  // at most 16,384 keys and 8,192 buckets: 192 KB
    const size_t smem = (size_t)cfg.n_coarse * sizeof(uint64_t) + 2 * sizeof(uint32_t) * ((size_t)1 << log2b);
    if (smem > 48 * 1024) {
        cudaError_t ea = cudaFuncSetAttribute(k_lem_lhs, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (ea != cudaSuccess) return ea;
    }
    // Each kernel a programmatic dependent of the one before it (the sampling
    // beside the update of the order before): 64 EEG-like channels, 20 orders,
    // 6.11 ms, plain launches 1 % more.
    cudaError_t e = launch_kernel(k_lem_lhs, dim3(B, 4), dim3(kLhsThreads), smem, st, pdl, cfg.n_coarse, log2b,
                                  cfg.box, cfg.seed, order, lb.cap, lb.cand, lb.ncand);
    const double inv_fs = 1.0 / fs;
    const size_t r_smem = sizeof(float) * (size_t)((L + 31) / 32 * 32);
    int n = cfg.n_coarse;
    for (int lev = 0; lev <= cfg.levels && e == cudaSuccess; ++lev) {
        int per = 1;
        if (lev > 0) {
            for (int a = 0; a < 4; ++a) per *= 2 * cfg.level[lev].radius[a] + 1;
            n = cfg.top_k * per;
        }
        const dim3 grid((n + kScreenCands - 1) / kScreenCands, B);
        e = launch_kernel(k_lem_screen, grid, dim3(kLemThreads), r_smem, st, pdl, lb.cap, lev, cfg.box, cfg.level[lev],
                          cfg.top_k, (const double *)lb.kept, (const int *)lb.nkept, lb.cand, lb.ncand, R, Lp, L,
                          inv_fs, lb.screen);
        if (e != cudaSuccess) break;
        e = launch_kernel(k_lem_pick, dim3(B), dim3(kPickThreads), sizeof(PickShared), st, pdl, lb.cap, cfg.top_k,
                          lev > 0 ? 1 : 0, (const double *)lb.cand, (const int *)lb.ncand, per, lb.nkept,
                          (const float2 *)lb.screen, R, Lp, L, inv_fs, lb.score, lb.kept, lb.kept_score);
    }
    return e;
}

int lem_kernels(const LemConfig &cfg) { return 3 + 2 * cfg.levels; }

}  // namespace act
