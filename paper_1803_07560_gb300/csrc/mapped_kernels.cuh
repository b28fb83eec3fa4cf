// mapped_kernels.cuh -- the range map of Sec. 4 (the infinite range of every
// coordinate taken to (-1, 1)) and Gaussian importance sampling as
// thread-per-sample FP64 kernels over the compiled lattice shapes, with their
// launchers.  Included by the shapes_*.cu files next to the box-sampler
// kernels.
//
//   transform_f64  persistent, thread per sample: Philox point y in the box,
//                  v_j = y_j / (1 - y_j^2), S_eff = S(v) - ln J with
//                  ln J = sum_j ln[(1 + y_j^2) / (1 - y_j^2)^2], weight,
//                  products and per-thread sums -> one FP64 record per chunk
//   gaussian_f64   the same with v = mean + F z, z standard normal from the
//                  unit point by the Box-Muller transform, S_eff = S(v) -
//                  |z|^2 / 2 and weight 0 outside the box (d <= 40)
//
// transform_f64 screens its samples in FP32 first, with a bound on the screen's
// own error for each sample, and evaluates in FP64 those that may carry
// weight (about one in twenty at 10x2 over all of R^20).  gaussian_f64
// evaluates every sample: under its proposal nine in ten carry weight.  Both
// are bound by GB300's FP64 pipe, so the FP64 work of an evaluation is kept
// small: one reciprocal per coordinate by Newton's iteration instead of a
// division, and one logarithm per sample for all of ln J.
#pragma once

#include "gauss_tables.h"
#include "integrand_kernels.cuh"

namespace bfi {

// 1/x within about an ulp: Newton's iteration for f(r) = 1/r - x,
// r <- r + r (1 - x r), which squares the relative error at each step, from
// the hardware's approximate reciprocal (PTX rcp.approx.ftz.f64).  Two steps
// take an error below 2^-20 to the rounding level.  x must be a positive
// normal number (here 1 - y^2 >= 2^-53); 0 gives NaN.
__device__ __forceinline__ double recip_newton(double x) {
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    double e = __fma_rn(-x, r, 1.0);
    r = __fma_rn(r, e, r);
    e = __fma_rn(-x, r, 1.0);
    return __fma_rn(r, e, r);
}

// ln of a product of factors >= 1, kept as p * 2^e with p brought back to
// [1, 2) by integer operations on its exponent field (no FP64 work), so that
// one logarithm serves the whole product.  renorm() after at most four
// factors below 2^255 each keeps p finite; an infinite or NaN p is left alone
// (its logarithm is then +inf or NaN, as the sum of the logarithms would be).
struct LogProduct {
    double p = 1.0;
    int e = 0;
    __device__ __forceinline__ void mul(double x) { p *= x; }
    __device__ __forceinline__ void renorm() {
        const int hi = __double2hiint(p);
        const int ex = (hi >> 20) & 0x7ff;
        if (ex != 0x7ff) {
            e += ex - 1023;
            p = __hiloint2double((hi & 0x000fffff) | 0x3ff00000, __double2loint(p));
        }
    }
    __device__ __forceinline__ double log_value() const {
        return fma(static_cast<double>(e), 0.6931471805599453, log(p));  // e ln 2 + ln p
    }
};

// ---------------------------------------------------------------------------
// FP32 screen of the range map, with bounds.  For a box inside [-1, 1]^d it
// returns S_lo and S_hi around the S_eff that the FP64 evaluation computes
// (u = 2^-24 below; "relative" errors are to first order):
//   * p = 1 + y = (1 + lo) + W u and m = 1 - y = (1 - hi) + W (1 - u) are sums
//     of non-negative terms, u from the word and 1 - u from its complement, so
//     both have a relative error of 4 u, r = 1 / (p m) of 11 u, and v = y r an
//     error of 17 u a, a = |v| + 1 >= r.
//   * The evaluation rounds y, and with it 1 -+ y, by up to 2^-52 (its last
//     bit, the rounding of W and of 1 + lo): v by 2^-51 r a, 8 u f a with
//     f = max(1, 2^-30 r of the sample's largest r).  Together |dv| <= eps a,
//     eps = 32 u f.
//   * The residual R = v_next + v (c_adv (v_r - v_l) + k1) - c_dif (v_r + v_l)
//     then has |dR| <= (2 eps + 8 u) T, T the sum of its terms' magnitudes with
//     a for |v|; the bound used is E = 2^-17 f T, 1.8 times that.
//     S between inv sum max(0, |R| - E)^2 and inv sum (|R| + E)^2.
//   * ln J = ln prod (1 + y^2) + 2 ln prod r, one logarithm for the first
//     product (at most 2^D) and one per Philox block for the second: 1e-3 f and
//     2^-15 of it cover the products' errors, y's rounding and lg2.approx's.
//     (Products of (1 + y^2) r^2 pass 2^128 where the r of a block pass 2^62
//     together, in boxes of width 2^-8 next to 1 about once in 2^20 samples.)
//   * A sample with an r beyond kMapMaxR (y within 2^-41 of +-1, one coordinate
//     in 2^41 over (-1, 1) and in 2^41 w over a slab of width w next to 1),
//     where these are no longer small, or with a product of r that overflows,
//     has no bound, [-inf, inf]: it is evaluated.
// The interval is a few thousandths wide for samples that matter, and it
// grows with the terms that cancel in a residual.  Overflows: residuals give
// S_lo = inf (true actions beyond 1e38) or NaN, which no comparison rejects,
// and S_hi = inf or NaN.
// ---------------------------------------------------------------------------
constexpr float kMapMaxR = 0x1p40f;

struct MapBox {
    float p0, m0, w;  // 1 + lo, 1 - hi, hi - lo
};

__device__ __forceinline__ MapBox map_box(double lo, double hi) {
    return MapBox{__double2float_rn(1.0 + lo), __double2float_rn(1.0 - hi), __double2float_rn(hi - lo)};
}

// The screen's premises: the box inside [-1, 1], and constants within float's
// range (an action that overflows is then beyond any window).
__device__ __forceinline__ bool map_box_screens(double lo, double hi) { return lo >= -1.0 && hi <= 1.0 && hi > lo; }
__device__ __forceinline__ bool map_consts_screen(const LatticeConst<float> &c) {
    return c.inv_2Dtau >= 1e-30f && c.inv_2Dtau <= 1e30f && fabsf(c.c_adv) <= 1e15f && fabsf(c.k1) <= 1e15f &&
           fabsf(c.neg_c_dif) <= 1e15f && c.half_mass2 <= 1e15f;
}

__device__ __forceinline__ float rcp_approx(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

template <int NX, int NT>
__device__ __forceinline__ void transform_screen(uint32_t x, const PhiloxPrefix *pre, const RoundKeys &rk,
                                                 const MapBox *box, const LatticeConst<float> &c, float &S_lo,
                                                 float &S_hi) {
    constexpr int D = NX * NT, NQ = (D + 3) / 4;
    const PhiloxFirst first = philox_first(x, pre[NQ].g);
    float v[D];
    float ln_r = 0.f, one_y2 = 1.f, r_max = 0.f;  // log2 prod r; prod (1 + y^2)
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        const uint4 b = philox_from_prefix(first, pre[q], rk);
        const uint32_t w4[4] = {b.x, b.y, b.z, b.w};
        float rs = 1.f;
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const int j = 4 * q + t;
            if (j < D) {
                const MapBox bx = box[j];
                const float u = fmaf(__uint2float_rn(w4[t]), 0x1p-32f, 0x1p-33f);
                const float u1 = fmaf(__uint2float_rn(~w4[t]), 0x1p-32f, 0x1p-33f);
                const float p = fmaf(u, bx.w, bx.p0), m = fmaf(u1, bx.w, bx.m0);
                const float r = rcp_approx(p * m), y = 0.5f * (p - m);
                v[j] = y * r;
                one_y2 *= fmaf(y, y, 1.f);
                rs *= r;
                r_max = fmaxf(r_max, r);
            }
        }
        ln_r += __log2f(rs);
    }
    const float ln_j = 0.69314718f * fmaf(2.f, ln_r, __log2f(one_y2));
    const float f = fmaxf(1.f, 0x1p-30f * r_max), eps = 0x1p-17f * f;
    const float a_adv = fabsf(c.c_adv), a_k1 = fabsf(c.k1), a_dif = fabsf(c.neg_c_dif);
    float low = 0.f, high = 0.f;
#pragma unroll
    for (int m = 0; m < NX; ++m) {
#pragma unroll
        for (int l = 0; l < NT; ++l) {
            const float here = v[m * NT + l], next = v[m * NT + (l + 1) % NT];
            const float right = v[((m + 1) % NX) * NT + l], left = v[((m + NX - 1) % NX) * NT + l];
            float R = fmaf(here, fmaf(c.c_adv, right - left, c.k1), next);
            R = fmaf(c.neg_c_dif, right + left, R);
            const float side = fabsf(right) + fabsf(left) + 2.f;
            float T = fmaf(fabsf(here) + 1.f, fmaf(a_adv, side, a_k1), fabsf(next) + 1.f);
            T = fmaf(a_dif, side, T);
            const float over = fmaf(eps, T, fabsf(R)), under = fmaxf(fmaf(-eps, T, fabsf(R)), 0.f);
            low = fmaf(under, under, low);
            high = fmaf(over, over, high);
        }
    }
    low *= c.inv_2Dtau;
    high *= c.inv_2Dtau;
    if (c.half_mass2 != 0.f) {
        float s_lo = 0.f, s_hi = 0.f;
#pragma unroll
        for (int j = 0; j < D; ++j) {
            const float a = fabsf(v[j]), e = 0.5f * fmaf(eps, a, eps), under = fmaxf(a - e, 0.f), over = a + e;
            s_lo = fmaf(under, under, s_lo);
            s_hi = fmaf(over, over, s_hi);
        }
        low = fmaf(c.half_mass2, s_lo, low);
        high = fmaf(c.half_mass2, s_hi, high);
    }
    S_lo = fmaf(low, 1.f - 0x1p-15f, -fmaf(ln_j, 1.f + 0x1p-15f, 1e-3f * f));
    S_hi = fmaf(high, 1.f + 0x1p-15f, -fmaf(ln_j, 1.f - 0x1p-15f, -1e-3f * f));
    if (r_max > kMapMaxR || !(ln_j < INFINITY)) {
        S_lo = -INFINITY;
        S_hi = INFINITY;
    }
}

// Floats as integers in the same order (NaN aside), for atomicMin.
__device__ __forceinline__ int order_f32(float x) {
    const int b = __float_as_int(x);
    return b ^ ((b >> 31) & 0x7fffffff);
}
__device__ __forceinline__ float unorder_f32(int b) { return __int_as_float(b ^ ((b >> 31) & 0x7fffffff)); }

// Reference action of a subvolume: the smallest S_hi among its first
// hint_samples(n_s) samples, or +inf where the screen is not to be used (its
// premises fail, or more than one in 256 of these samples has no bound, or the
// interval of that sample is wider than kMapResolved, the margin that moves a
// shift, as in slabs close to +-1): every sample of the subvolume is then
// evaluated.  So it is where the screen gains nothing: where more than 15 in 16
// of the first 256 lie within the window of the reference, or more than half
// while the interval is wider than 8, which leaves most threads open.
// Measured on GB300 at nu = 6 (2^20 to 2^24 samples, intervals of 0.1 to 8):
// 10x2 20.4 ms at a limit of 0.05 against 0.80 ms at 1, 4 and 16; 32x2 4.95 ms
// at 0.05, 4.75 at 4, 0.81 at 16.  At 2x2, 300 x 2000 samples screened and
// evaluated throughout: [-1, 1]^4 with D = 4^8 309 and 269 us; [1 - 2^-20, 1]^4
// with D = 4^25, all within the window, 390 and 266; at widths of 4 to 8 and
// three in four samples 279 and 283.  One CTA per subvolume.
constexpr float kMapResolved = 16.f;

template <int NX, int NT>
__global__ void __launch_bounds__(kBlock) hint_transform(const IntegrandArgs args, const LatticeConst<float> lc,
                                                         const RoundKeys rk) {
    constexpr int D = NX * NT, NQ = (D + 3) / 4;
    __shared__ int s_min, s_low, s_bad;
    __shared__ unsigned s_unbound, s_near;
    __shared__ MapBox s_map[D];
    __shared__ PhiloxPrefix s_pre[NQ + 1];
    const int64_t s = blockIdx.x;
    const int tid = threadIdx.x;
    if (tid == 0) {
        s_min = s_low = order_f32(INFINITY);
        s_bad = map_consts_screen(lc) ? 0 : 1;
        s_unbound = s_near = 0u;
    }
    __syncthreads();
    const uint32_t sid = args.sub_id ? args.sub_id[s] : static_cast<uint32_t>(s);
    if (tid < NQ) s_pre[tid] = philox_prefix(tid, 0u, sid, rk);
    if (tid == NQ) s_pre[NQ].g = philox_word0(0u, rk);
    if (tid < D) {
        const double lo = args.lo[s * D + tid], hi = args.hi[s * D + tid];
        s_map[tid] = map_box(lo, hi);
        if (!map_box_screens(lo, hi)) s_bad = 1;
    }
    __syncthreads();
    const uint32_t n = static_cast<uint32_t>(hint_samples(args.samples[s]));
    float mn = INFINITY, ln = INFINITY, lo_first = INFINITY;
    for (uint32_t k = tid; k < n; k += kBlock) {
        float lo, hi;
        transform_screen<NX, NT>(k, s_pre, rk, s_map, lc, lo, hi);
        if (k == static_cast<uint32_t>(tid)) lo_first = lo;
        mn = fminf(mn, hi);
        if (lo == -INFINITY)
            atomicAdd(&s_unbound, 1u);
        else
            ln = fminf(ln, lo);
    }
    // a warp's result first: 256 atomics on one word would take longer than a short hint's samples
    const int w_min = __reduce_min_sync(0xffffffffu, order_f32(mn)), w_low = __reduce_min_sync(0xffffffffu, order_f32(ln));
    if ((tid & 31) == 0) {
        atomicMin(&s_min, w_min);
        atomicMin(&s_low, w_low);
    }
    __syncthreads();
    const float best = unorder_f32(s_min), width = best - unorder_f32(s_low);
    const unsigned near = __ballot_sync(0xffffffffu, !(lo_first > __fadd_ru(best, args.skip_window)));
    if ((tid & 31) == 0) atomicAdd(&s_near, __popc(near));
    __syncthreads();
    if (tid == 0) {
        const unsigned of = min(n, static_cast<uint32_t>(kBlock));
        const bool bad = s_bad || 256u * s_unbound > n || !(width <= kMapResolved) || 16u * s_near > 15u * of ||
                         (width > 8.f && 2u * s_near > of);
        args.hint[s] = bad ? INFINITY : best;
    }
}

// ---------------------------------------------------------------------------
// One CTA processes chunk blockIdx.x, then the chunks next_chunk hands it;
// thread t screens samples first + t, first + t + B, ... of the chunk.  Those
// whose S_lo is within the negligible-weight window of the reference (the
// hint, then the smallest action evaluated) go to the warp's queue and are
// evaluated in FP64, 32 at a time: the Philox words, the point y = lo +
// (hi - lo) u (the FP64 point of the box sampler) and 1 - y^2 = (1 - y)(1 + y)
// are those of the definition; v_j = y_j r_j with r_j = 1 / (1 - y_j^2), and
// J_j = (1 + y_j^2) r_j^2 joins the running product.
//
// The record's shift is defined by the samples alone, not by which of them
// are evaluated or where: every thread's shift drops from +inf to its first
// sample's S_eff and from then on only to a sample more than kRescaleMargin
// below it, and the record has the smallest of the threads' shifts.  The
// screen follows each thread's shift as an interval [m_lo, m_hi] with the
// sample k_m that set it; a sample that may or may not have moved it leaves
// the interval wide ('open') until one lies surely below both ends.  At the
// chunk's end the threads whose interval reaches the smallest m_hi decide:
// k_m is as a rule among the evaluated samples (the window is wider than the
// margin), whose S_eff was kept, and is evaluated now where the whole chunk
// lies outside the window of another chunk's reference.  An open thread goes
// through its samples again from k_m on, with the exact shift in hand, and
// evaluates in FP64 those that may lie below it by the margin; its warp's
// other open threads do so beside it, and the other warps wait.  (The whole
// CTA used to take one open thread after another.  Measured on GB300 at 2x2,
// where every sample's evaluation takes 158 us for 8 x 2^15 samples and 265 us
// for 300 x 2000: [1 - 2^-16, 1]^4 with D = 4^16, whose intervals are 13 wide,
// 5414 -> 231 us and, of 300 x 2000, 392 us now.)
// A chunk with no finite S_eff records m = +inf and zero sums.
//
// Where the hint is +inf every sample goes through the queue, a warp's row at
// once, so that lane l evaluates its own sample and its sums' shift is the
// thread's shift.
//
// What bounds it: the FP64 pipe takes a warp instruction every 64 cycles per
// scheduler, ~590 of them an evaluation, against ~1000 instructions of the
// screen per row of 32 samples; two CTAs per SM let one's evaluations run
// under the other's screen (lattices over 32 sites hold the FP64 field of an
// evaluation in over 128 registers: one CTA; up to 4 sites three fit with 80,
// and an open thread's shift lies in shared memory to keep it so: 2x2, 3000 x
// 60 samples take 200 us, 235 at two CTAs).
//
// Measured on GB300 (whole pass, against the kernel that evaluated every
// sample; nu = 1, [-1, 1]^d bisected): 10x2, 256 x 2^16 samples 19.55 ->
// 1.67 ms; one volume of 2^22 samples at 4x2 5.83 -> 1.00 ms (a third of its
// samples carry weight), at 8x4 10.8 -> 0.55 ms; 500 x 524 at 10x2 3.06 ->
// 0.46 ms.
// ---------------------------------------------------------------------------
template <int NX, int NT, int BLOCK>
__global__ void __launch_bounds__(BLOCK, NX *NT <= 32 ? 2 : 1)
    transform_f64(const IntegrandArgs args, const LatticeConst<double> lc, const LatticeConst<float> lcf,
                  const RoundKeys rk) {
    constexpr int D = NX * NT;
    constexpr int R = NX / 2 + 1;
    constexpr int K = sum_count(R);
    constexpr int NQ = (D + 3) / 4;
    constexpr int WARPS = BLOCK / 32;
    __shared__ ChunkShared<BLOCK> sh;
    __shared__ double s_lo[D], s_w[D], s_S[BLOCK];
    __shared__ MapBox s_map[D];
    __shared__ PhiloxPrefix s_pre[NQ + 1];
    __shared__ double s_sums[K * BLOCK];
    __shared__ uint32_t s_queue[WARPS][kQueueCap], s_km[BLOCK], s_known[BLOCK];
    __shared__ long long s_shift;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned lt = (1u << lane) - 1u;
    uint32_t *queue = s_queue[warp];
    SmemSums<double, K, BLOCK> acc{s_sums + tid};
    constexpr uint32_t kNone = 0xffffffffu;  // no sample (offsets in a chunk are below 2^31)

    for (int64_t c = blockIdx.x; c < args.nchunks; c = next_chunk(args, c, &sh.next)) {
        const ChunkView v = chunk_view(args, c, D);
        const float hint = args.hint[v.s];
        const bool direct = !(hint < INFINITY);
        if (tid < D) {
            s_lo[tid] = v.lo[tid];
            s_w[tid] = v.hi[tid] - v.lo[tid];
            s_map[tid] = map_box(v.lo[tid], v.hi[tid]);
        }
        chunk_prefixes<D>(v, rk, s_pre);
        if (tid == 0) {
            sh.evaluated = 0u;
            sh.min_bits = order_f32(hint);
            s_shift = order_f64(INFINITY);
        }
        s_km[tid] = s_known[tid] = kNone;
        acc.zero();
        __syncthreads();

        double m_acc = INFINITY;                    // shift of this thread's sums
        float m_ref = hint, m_lo = INFINITY, m_hi = INFINITY;
        bool open = false;
        unsigned n_eval = 0;
        int count = 0;
        const uint32_t cnt = static_cast<uint32_t>(v.cnt), xb = static_cast<uint32_t>(v.first);
        const uint32_t nrows = (cnt + BLOCK - 1) / BLOCK;
        bool ask = false;                           // this thread decides and its k_m has not been evaluated
        bool walk = false;                          // this thread decides and is open: its shift is followed, in
                                                    // s_S, from sample s_km on (or from its first)
        // rows 0 .. nrows - 1; then the samples left in the queues; then the k_m that decide but were outside the
        // window; then the open threads' rows again, warp by warp
        for (uint32_t row = 0;;) {
            const bool again = row > nrows + 1;
            const uint32_t k = (again ? row - nrows - 2 : row) * BLOCK + tid;
            const bool follows = again && walk && k < cnt && (s_km[tid] == kNone || k >= s_km[tid]);
            uint32_t k_eval = 0u;
            float lo = -INFINITY, hi = INFINITY;
            if (row < nrows ? k < cnt && !direct : follows && s_S[tid] < INFINITY)
                transform_screen<NX, NT>(xb + k, s_pre, rk, s_map, lcf, lo, hi);
            bool evaluate = false;
            if (row < nrows) {
                bool cand = false;
                if (k < cnt) {
                    cand = true;
                    if (!direct) {
                        cand = !(lo > __fadd_ru(m_ref, args.skip_window));
                        const float slack = kRescaleMargin + 0x1p-20f * fabsf(m_lo);
                        if (hi < m_lo - slack || (m_lo == INFINITY && hi < INFINITY)) {
                            m_lo = lo;
                            m_hi = hi;
                            open = !(lo > -INFINITY);
                            s_km[tid] = k;
                        } else if (!(m_hi < INFINITY && lo >= m_hi - kRescaleMargin + 0x1p-20f * fabsf(m_hi))) {
                            m_lo = lo < m_lo ? lo : (lo == lo ? m_lo : -INFINITY);
                            open = true;
                        }
                    }
                }
                count = enqueue(queue, count, cand, k, lt);
                evaluate = count >= 32;
                if (evaluate) k_eval = queue[lane];
            } else if (row == nrows) {
                if (direct) {  // fewer than a row: the lanes' own samples
                    evaluate = lane < count;
                    if (evaluate) k_eval = queue[lane];
                } else {       // gathered in warp order and evaluated in as few warps as possible
                    uint32_t *flat = &s_queue[0][0];
                    const uint32_t mine = lane < count ? queue[lane] : 0u;
                    if (lane == 0) sh.left[warp] = count;
                    __syncthreads();
                    int off = 0, total = 0;
#pragma unroll
                    for (int w = 0; w < WARPS; ++w) {
                        const int c_w = sh.left[w];
                        off += w < warp ? c_w : 0;
                        total += c_w;
                    }
                    if (lane < count) flat[off + lane] = mine;
                    __syncthreads();
                    evaluate = tid < total;
                    if (evaluate) k_eval = flat[tid];
                }
            } else if (row == nrows + 1) {
                evaluate = ask;
                if (ask) k_eval = s_km[tid];
            } else {
                const float m = __double2float_ru(s_S[tid]);
                evaluate = follows && !(lo >= m - kRescaleMargin + 0x1p-20f * fabsf(m));
                k_eval = k;
            }
            if (evaluate) {
                const PhiloxFirst first = philox_first(xb + k_eval, s_pre[NQ].g);
                double u[D];
                LogProduct jac;
#pragma unroll
                for (int q = 0; q < NQ; ++q) {
                    const uint4 b = philox_from_prefix(first, s_pre[q], rk);
                    const uint32_t w4[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
                    for (int t = 0; t < 4; ++t) {
                        const int j = 4 * q + t;
                        if (j < D) {
                            const double y = Coord<double>::map(w4[t], s_lo[j], s_w[j]);
                            const double r = recip_newton((1.0 - y) * (1.0 + y));
                            u[j] = y * r;
                            jac.mul(fma(y, y, 1.0) * r * r);
                            if (j % 2 == 1 || j == D - 1) jac.renorm();
                        }
                    }
                }
                const double S = action<NX, NT, double>(u, lc) - jac.log_value();
                if (row <= nrows) {
                    m_ref = fminf(m_ref, __double2float_ru(S));
                    const uint32_t owner = k_eval % BLOCK;
                    if (!direct && s_km[owner] == k_eval) {  // one evaluation of each sample: no two threads write
                        s_S[owner] = S;
                        s_known[owner] = k_eval;
                    }
                    double Q[R];
                    products<NX, NT, double>(u, Q);
                    if (S < m_acc - kRescaleMargin) {  // the first sample, then rarely
                        rescale<double, K, R, BLOCK>(acc, exp(S - m_acc));
                        m_acc = S;
                    }
                    accumulate<K, R, BLOCK>(acc, exp(m_acc - S), Q);
                    ++n_eval;
                } else if (!again || S < s_S[tid] - kRescaleMargin) {
                    s_S[tid] = S;
                }
            }
            if (row < nrows) {
                if (evaluate) {
                    count = dequeue32(queue, count);
                    m_ref = unorder_f32(__reduce_min_sync(0xffffffffu, order_f32(m_ref)));
                }
                if (++row % kShareRows == 0 && row < nrows) {
                    atomicMin(&sh.min_bits, order_f32(m_ref));
                    __syncthreads();
                    m_ref = unorder_f32(sh.min_bits);
                    __syncthreads();
                }
                continue;
            }
            if (direct) break;
            if (row == nrows) {
                if (tid == 0) sh.min_bits = order_f32(INFINITY);
                __syncthreads();
                atomicMin(&sh.min_bits, order_f32(m_hi));
                __syncthreads();
                const bool decides = static_cast<uint32_t>(tid) < cnt && m_lo <= unorder_f32(sh.min_bits);
                const bool known = !open && s_known[tid] == s_km[tid];
                if (decides && known) atomicMin(&s_shift, order_f64(s_S[tid]));
                ask = decides && !open && !known;
                walk = decides && open;
                if (walk) s_S[tid] = INFINITY;
                if (__syncthreads_or(ask)) {
                    row = nrows + 1;
                    continue;
                }
            } else if (row == nrows + 1) {
                if (ask) atomicMin(&s_shift, order_f64(s_S[tid]));
            }
            // the walk: no barrier until every warp has left the loop
            const uint32_t from = s_km[tid] == kNone ? 0u : s_km[tid] / BLOCK;
            row = again ? row + 1 : nrows + 2 + __reduce_min_sync(0xffffffffu, walk ? from : nrows);
            if (row < 2 * nrows + 2) continue;
            if (walk) atomicMin(&s_shift, order_f64(s_S[tid]));  // +inf moves nothing
            break;
        }
        add_evaluated(args.stats, n_eval, &sh.evaluated);
        if (direct) {
            chunk_record<double, K, R, BLOCK>(acc, m_acc, n_eval > 0, sh.f, &sh.mb, sh.left, args.partials + c * (K + 2), v.cnt);
        } else {
            __syncthreads();
            if (tid == 0) sh.mb = unorder_f64(s_shift);
            __syncthreads();
            chunk_record<double, K, R, BLOCK, true>(acc, m_acc, n_eval > 0, sh.f, &sh.mb, sh.left,
                                                    args.partials + c * (K + 2), v.cnt);
        }
    }
}

// ---------------------------------------------------------------------------
// Box-Muller pairs from words, by tables and short Taylor polynomials.  CUDA's
// log, sqrt and sincospi took over half of the Gaussian kernel's FP64
// instructions (about 70 of them a pair, on a pipe of 2 lanes per SM and
// clock); their arguments are one 33-bit number each, so a table by a few
// leading bits leaves little for a polynomial: 36 a pair.
//
//   t = -2 ln u, u = (w + 1/2) 2^-32 = m 2^e, m in [3/4, 3/2): with c a 20-bit
//     approximation of 1/m from the 7 leading bits, z = m c - 1 is exact,
//     |z| <= 2^-8, and t = -2 e ln 2 + 2 ln c - 2 ln(1 + z), the last by its
//     Taylor polynomial of degree 7 (remainder below 2^-58 z).  c = 1 next to
//     m = 1, so t keeps its relative accuracy as u -> 1.
//   r = sqrt(t): one Newton step for 1/sqrt(t) from the hardware's
//     approximation (PTX rsqrt.approx.ftz.f64) and one for the root.
//   cos, sin of 2 pi u: the angle is that of the nearest of 1024 points of the
//     circle plus x, |x| <= pi/1024; Taylor polynomials of degree 5 and 4
//     (remainders below 2^-61), then the angle sum.
// Table entries are pairs (hi, lo): the small terms are summed first, so a
// result carries about one rounding.  Measured against 113-bit arithmetic over
// 2^21 pairs, near the ends of u1 and the axes among them, the error of z over
// r in units of 2^-53: at most 2.77, rms 0.512; with CUDA's functions 2.77 and
// 0.534.
// ---------------------------------------------------------------------------
// constant data of each translation unit that includes this file
static __device__ const tables::Octant kOctant = tables::make_octant();
static __device__ const tables::Logs kLogs = tables::make_logs();

struct __align__(16) Quad {
    double x, y, z, w;
};

struct GaussTables {
    Quad log_c[128];         // (c, 2 ln c as hi, lo) of the intervals of m
    double2 log_e[34];       // 2 k ln 2, k = -e
    Quad circle[1024];       // (cos, sin, and their lower parts) of 2 pi j / 1024
};

// Filled by the CTA (at least 129 threads); the caller synchronises.
__device__ __forceinline__ void fill_gauss_tables(GaussTables &t) {
    const int i = threadIdx.x;
    if (i < 128) t.log_c[i] = Quad{kLogs.c[i], kLogs.hi[i], kLogs.lo[i], 0.0};
    if (i < 34) t.log_e[i] = make_double2(kLogs.k_hi[i], kLogs.k_lo[i]);
    if (i <= 128) {
        const double c = kOctant.c[i], s = kOctant.s[i], cl = kOctant.c_lo[i], sl = kOctant.s_lo[i];
#pragma unroll
        for (int o = 0; o < 8; ++o) {  // the first octant, the others by symmetry
            if (i == (o % 2 == 0 ? 128 : 0)) continue;
            const bool even = o % 2 == 0;
            const double a = even ? c : s, b = even ? s : c, al = even ? cl : sl, bl = even ? sl : cl;
            const int q = o / 2, j = even ? o * 128 + i : (o + 1) * 128 - i;
            t.circle[j] = q == 0   ? Quad{a, b, al, bl}
                          : q == 1 ? Quad{-b, a, -bl, al}
                          : q == 2 ? Quad{-a, -b, -al, -bl}
                                   : Quad{b, -a, bl, -al};
        }
    }
}

// z0 = r cos(2 pi u2), z1 = r sin(2 pi u2) and r^2 = -2 ln u1 = z0^2 + z1^2.
__device__ __forceinline__ void box_muller_words(uint32_t w1, uint32_t w2, const GaussTables &tab, double &z0,
                                                 double &z1, double &r2) {
    const double u = unit_f64(w1);
    const int hi = __double2hiint(u), d = hi - 0x3fe80000, e = d >> 20;
    const Quad c = tab.log_c[(d >> 13) & 127];
    const double2 l2 = tab.log_e[-e];
    const double z = fma(__hiloint2double(hi - (e << 20), __double2loint(u)), c.x, -1.0);
    double q = fma(z, -2.0 / 7.0, 1.0 / 3.0);
    q = fma(z, q, -2.0 / 5.0);
    q = fma(z, q, 0.5);
    q = fma(z, q, -2.0 / 3.0);
    q = fma(z, q, 1.0);
    const double t = (l2.x + c.y) + fma(z, -2.0, fma(z * z, q, l2.y + c.z));
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(t));
    double g = t * y, h = __hiloint2double(__double2hiint(y) - 0x00100000, __double2loint(y));  // y / 2
    const double f = fma(-g, h, 0.5);
    g = fma(g, f, g);
    h = fma(h, f, h);
    const double r = fma(fma(-g, g, t), h, g);
    // angle: 1024 points of 2^22 words each; x = 2 pi 2^-32 (k + 1/2), k = w2 - nearest, made a double by its bits:
    // 2^52 + 2^31 + k, less 2^52 + 2^31
    const uint32_t j = (w2 + 0x200000u) >> 22;
    const uint32_t k = (w2 - (j << 22)) ^ 0x80000000u;
    const double x = fma(__hiloint2double(0x43300000, static_cast<int>(k)) - 4503601774854144.0, 1.4629180792671596e-9,
                         0.5 * 1.4629180792671596e-9);
    const Quad p = tab.circle[j & 1023u];
    const double x2 = x * x;
    const double sx = fma(x * x2, fma(x2, 1.0 / 120.0, -1.0 / 6.0), x), cx1 = x2 * fma(x2, 1.0 / 24.0, -0.5);
    z0 = r * (p.x + fma(-p.y, sx, fma(p.x, cx1, p.z)));
    z1 = r * (p.y + fma(p.x, sx, fma(p.y, cx1, p.w)));
    r2 = t;
}

// x >= lo and x < hi by integers that order as the doubles do: no FP64
// instruction.  Bounds that are zero take the key of -0, which both zeros
// reach; NaN bounds admit nothing.
__device__ __forceinline__ long long bound_key(double b) {
    return b != b ? 0x7fffffffffffffffll : order_f64(b == 0.0 ? -0.0 : b);
}

// ---------------------------------------------------------------------------
// Gaussian importance sampling, thread per sample (d <= kGaussThreadMaxD):
// z_{2p}, z_{2p+1} by Box-Muller from u_{2p}, u_{2p+1} for the unit point u (the
// box plays no part in drawing; for odd d the pair of z_{d-1} takes word d of
// the last Philox block), v = mean + F z, S_eff = S(v) - |z|^2 / 2, and
// weight 0 outside the box
// [lo, hi).  The rest of 1/q (the record's log-volume (d/2) ln 2 pi +
// ln |det F|) is set by the merge.  F, held transposed in shared memory
// (column j of F contiguous, every thread reading the same word), is applied
// column by column as each z_j is drawn, so z is never stored; for an upper
// triangular F (TRI, the proposal bfi_gaussian_proposal returns) column j
// stops at row j.  Samples outside the box are counted in n and skip the
// action; the kernel counts the evaluated (inside) samples in stats.
//
// What bounds it: the FP64 pipe, which takes a warp instruction every 64
// cycles per scheduler; two warps per scheduler keep it busy, so the kernel is
// compiled for one CTA per SM with all the registers a thread may have.  At
// 10x2 about 860 FP64 instructions a sample: 360 for the ten pairs, 210 for
// F z, 120 for the action, 111 for the products, the rest for the weight and
// the sums (869 counted, the pipe 91% busy; 1300 before the tables, the sums
// by FMA and the box test off the pipe).  Measured on GB300, 2^22 samples at
// 10x2: 9.94 -> 6.72 ms.
// ---------------------------------------------------------------------------
constexpr int kGaussThreadMaxD = 40;

template <int NX, int NT, int BLOCK, bool TRI>
__global__ void __launch_bounds__(BLOCK, 1) gaussian_f64(const IntegrandArgs args, const LatticeConst<double> lc,
                                                         const RoundKeys rk, const double *mean,
                                                         const double *factor) {
    constexpr int D = NX * NT;
    constexpr int R = NX / 2 + 1;
    constexpr int K = sum_count(R);
    constexpr int NQ = (D + 3) / 4;
    static_assert(D <= kGaussThreadMaxD, "the thread-per-sample Gaussian kernel holds v in registers");
    __shared__ ChunkShared<BLOCK> sh;
    __shared__ GaussTables s_tab;
    __shared__ double s_ft[D * D];  // s_ft[j D + r] = F[r][j]
    __shared__ double s_mean[D];
    __shared__ long long s_lo[D], s_hi[D];
    __shared__ PhiloxPrefix s_pre[NQ + 1];
    __shared__ double s_sums[K * BLOCK];
    const int tid = threadIdx.x;
    SmemSums<double, K, BLOCK> acc{s_sums + tid};
    fill_gauss_tables(s_tab);
    for (int k = tid; k < D * D; k += BLOCK) s_ft[(k % D) * D + k / D] = factor[k];
    for (int k = tid; k < D; k += BLOCK) s_mean[k] = mean ? mean[k] : 0.0;

    for (int64_t c = blockIdx.x; c < args.nchunks; c = next_chunk(args, c, &sh.next)) {
        const ChunkView v = chunk_view(args, c, D);
        if (tid < D) {
            const double lo = v.lo[tid], hi = v.hi[tid];
            s_lo[tid] = bound_key(hi != hi ? hi : lo);
            s_hi[tid] = bound_key(hi);
        }
        chunk_prefixes<D>(v, rk, s_pre);
        if (tid == 0) sh.evaluated = 0u;
        acc.zero();
        __syncthreads();

        double m_acc = INFINITY;
        unsigned n_eval = 0;
        for (uint64_t k = tid; k < v.cnt; k += BLOCK) {
            const PhiloxFirst first = philox_first(static_cast<uint32_t>(v.first + k), s_pre[NQ].g);
            // F is read again for every sample: hidden from the compiler, which would otherwise carry as much of it
            // as it can in registers and spill the rest
            const double *ft = s_ft;
            asm volatile("" : "+l"(ft));
            double u[D];
#pragma unroll
            for (int r = 0; r < D; ++r) u[r] = s_mean[r];
            double zz = 0.0;
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                const uint4 b = philox_from_prefix(first, s_pre[q], rk);
                const uint32_t w4[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
                for (int t = 0; t < 4; t += 2) {
                    const int j = 4 * q + t;
                    if (j < D) {
                        double zp[2], r2;
                        box_muller_words(w4[t], w4[t + 1], s_tab, zp[0], zp[1], r2);
                        zz = j + 1 < D ? zz + r2 : fma(zp[0], zp[0], zz);
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            if (j + e < D) {
                                const double z = zp[e];
#pragma unroll
                                for (int r = 0; r < (TRI ? j + e + 1 : D); ++r)
                                    u[r] = fma(ft[(j + e) * D + r], z, u[r]);
                            }
                        }
                    }
                }
            }
            bool inside = true;
#pragma unroll
            for (int r = 0; r < D; ++r) {
                const long long key = order_f64(u[r]);
                inside = inside && key >= s_lo[r] && key < s_hi[r];
            }
            if (!inside) continue;  // weight 0
            const double S = action<NX, NT, double>(u, lc) - 0.5 * zz;
            double Q[R];
            products<NX, NT, double>(u, Q);
            if (S < m_acc - kRescaleMargin) {
                rescale<double, K, R, BLOCK>(acc, exp(S - m_acc));
                m_acc = S;
            }
            accumulate<K, R, BLOCK>(acc, exp(m_acc - S), Q);
            ++n_eval;
        }
        add_evaluated(args.stats, n_eval, &sh.evaluated);
        chunk_record<double, K, R, BLOCK>(acc, m_acc, n_eval > 0, sh.f, &sh.mb, sh.left, args.partials + c * (K + 2), v.cnt);
    }
}

template <int NX, int NT>
cudaError_t launch_gaussian(const IntegrandArgs &args, const LatticeParams &p, const MapArgs &m, bool upper,
                            uint32_t seed, uint32_t job, int grid, cudaStream_t st) {
    const RoundKeys rk = make_round_keys(seed, job);
    if (upper)
        gaussian_f64<NX, NT, kBlock, true><<<grid, kBlock, 0, st>>>(args, make_const<double>(p), rk, m.mean, m.factor);
    else
        gaussian_f64<NX, NT, kBlock, false><<<grid, kBlock, 0, st>>>(args, make_const<double>(p), rk, m.mean, m.factor);
    return cudaGetLastError();
}

template <int NX, int NT>
cudaError_t occupancy_gaussian(int, int, int *blocks_per_sm) {
    int a = 0, b = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, gaussian_f64<NX, NT, kBlock, true>, kBlock, 0);
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, gaussian_f64<NX, NT, kBlock, false>, kBlock, 0);
    *blocks_per_sm = a < b ? a : b;
    return e;
}

// The Gaussian entries of the shape table: null above kGaussThreadMaxD (those
// shapes use generic_mapped<2>).
template <int NX, int NT>
constexpr GaussLauncher gaussian_entry() {
    if constexpr (NX * NT <= kGaussThreadMaxD) return launch_gaussian<NX, NT>;
    else return nullptr;
}
template <int NX, int NT>
constexpr OccupancyQuery gaussian_occupancy_entry() {
    if constexpr (NX * NT <= kGaussThreadMaxD) return occupancy_gaussian<NX, NT>;
    else return nullptr;
}

template <int NX, int NT>
cudaError_t launch_transform(const IntegrandArgs &args, const LatticeParams &p, uint32_t seed, uint32_t job, int grid,
                             cudaStream_t st) {
    const RoundKeys rk = make_round_keys(seed, job);
    hint_transform<NX, NT><<<static_cast<unsigned>(args.nsub), kBlock, 0, st>>>(args, make_const<float>(p), rk);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    transform_f64<NX, NT, kBlock><<<grid, kBlock, 0, st>>>(args, make_const<double>(p), make_const<float>(p), rk);
    return cudaGetLastError();
}

template <int NX, int NT>
cudaError_t occupancy_transform(int, int, int *blocks_per_sm) {
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, transform_f64<NX, NT, kBlock>, kBlock, 0);
}

}  // namespace bfi
