// integrand.cu -- the hot path of the Monte Carlo evaluation of the lattice
// Burgers functional integral (Honkonen & Honkonen, arXiv:1803.07560,
// Eq. (Gen2), Sec. 3 and Sec. 4) as sm_103a kernels:
//
//   integrand_f64 / integrand_f32
//                  persistent, thread-per-sample: Philox points -> action ->
//                  shifted weight -> products -> per-thread sums; then a
//                  warp / block merge of shifted records into one partial
//                  record per chunk of samples
//   hint_f32       per-subvolume reference action (the smallest FP32 action
//                  of the first samples), the starting point of both kernels
//   merge_records  FP64 merge of each subvolume's chunk records into its slot,
//                  then of all slots into Z, C(r) and errors
//
// Every reduction has a fixed order, so results are bitwise reproducible and do
// not depend on what else runs on the device.
#include "integrand_kernels.cuh"

#include <algorithm>
#include <climits>
#include <cmath>

namespace bfi {
// ---------------------------------------------------------------------------
// FP64 merge of the chunk records into subvolume slots and of the slots into
// the totals, in one kernel.
//
// What bounds it: latency and the FP64 pipe (2 lanes per SM and clock: a warp
// instruction takes the SM's pipe for 16 cycles however few lanes work), not
// bytes.  So a subvolume's records are merged by one warp (by many, 32 chunks
// each, where it has more than kMergeWhole), warps spread over the SMs; the
// factors of 32 chunks are computed at once, one per lane; the sums stay in
// registers with eight records' loads in flight; every logarithm, exponential
// and division that the totals need of a subvolume is done by its own warp,
// all SMs at work; and the CTA that finishes last is left with additions and
// a multiplication by a power of two per subvolume, what is the same for all
// threads done by one warp.
//
// Measured on GB300 (kernel time; before: two kernels, one warp per subvolume
// that kept its sums in global memory, and one CTA for all of the totals'
// arithmetic): one volume of 1024 chunks at 4x2 713 -> 25 us, of 4096 chunks
// at 10x2 4078 -> 31 us; 3 subvolumes of 41 chunks 123 -> 21 us; 1024 of 5 or
// 6 chunks at 10x2 139 -> 37 us; 256 of 16 chunks at 64x8 245 -> 37 us.
// ---------------------------------------------------------------------------
// CTAs that the tasks spread over before a CTA takes a second one: one per SM,
// since a CTA's warps share the SM's FP64 pipe.
constexpr int kMergeSpread = 152;
constexpr int kMergeThreads = 512, kMergeWarps = kMergeThreads / 32;
constexpr int kFarLog = (1023 + 60) << 20;  // upper word of 2^60 (see finish_subvolume)

__device__ __forceinline__ double warp_sum_f64(double v) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    return v;
}

// x == +0, off the FP64 pipe; 2^e (0 below the normal range, e <= 0).
__device__ __forceinline__ bool is_zero(double x) { return __double_as_longlong(x) == 0; }
__device__ __forceinline__ double pow2(int e) { return e < -1022 ? 0.0 : __hiloint2double((1023 + e) << 20, 0); }

// Sums of the records at(0) .. at(count - 1) at their smallest shift, in FP64:
// lane t adds sums t, t + 32, ... (four running sums of every fourth record,
// then those in order) and hands them to put(k, sum); returns the shift on
// every lane.
template <typename At, typename Put>
__device__ __forceinline__ double merge_list(int64_t count, int R, At at, Put put) {
    const int lane = threadIdx.x & 31, K = sum_count(R);
    // the smallest shift, by the integers that order as the doubles do (no shift is NaN): off the FP64 pipe
    long long lowest = order_f64(INFINITY);
    for (int64_t i = lane; i < count; i += 32) lowest = min(lowest, order_f64(__ldcg(at(i) + 1)));
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) lowest = min(lowest, __shfl_xor_sync(0xffffffffu, lowest, off));
    const double m = unorder_f64(lowest);
    for (int k0 = 0; k0 < K; k0 += 32) {
        const int k = k0 + lane;
        const bool mine = k < K, sq = mine && second_order(k, R);
        double acc[4] = {0.0, 0.0, 0.0, 0.0};
        for (int64_t c0 = 0; c0 < count; c0 += 32) {
            const int cnt = static_cast<int>(min(static_cast<int64_t>(32), count - c0));
            double f = 0.0, f2 = 0.0;  // of record c0 + lane; 0: no evaluated samples in it
            if (lane < cnt) {
                const double mc = __ldcg(at(c0 + lane) + 1);
                f = order_f64(mc) == order_f64(INFINITY) ? 0.0 : (order_f64(mc) == lowest ? 1.0 : exp(m - mc));
                f2 = f * f;
            }
            const unsigned weighted = __ballot_sync(0xffffffffu, __double_as_longlong(f) != 0);
            for (int i0 = 0; i0 < cnt; i0 += 8) {
                double v[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) v[i] = mine && i0 + i < cnt ? __ldcg(at(c0 + i0 + i) + 2 + k) : 0.0;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const double fi = __shfl_sync(0xffffffffu, f, i0 + i), f2i = __shfl_sync(0xffffffffu, f2, i0 + i);
                    if ((weighted >> (i0 + i)) & 1u) acc[i % 4] = fma(v[i], sq ? f2i : fi, acc[i % 4]);
                }
            }
        }
        __syncwarp();
        if (mine) put(k, (acc[0] + acc[1]) + (acc[2] + acc[3]));
    }
    return m;
}

// The slot of a subvolume (its sums are in slot[3 ...], unscaled products
// Q_r = d P_r) and what the totals need of it:
//   ls = log V - log n - m = k ln 2 + ln t, so that f_s / 2^kmax =
//   t 2^(k - kmax) once the largest k is known;
//   f_buf[s] = t, f_buf[nsub + s] = t^2 / (n - 1), and, in the place of the
//   subvolume's first chunk record, k, V_Z, V_N(r) and Cov(r) without f.
// k is an integer in a double: t lies in [2^-1/2, 2^1/2], but for |ls| near 2^60,
// as tiny D can make it, where k's own rounding leaves it in e^+-200.  From there
// on two ls are equal or further apart than any weight, so t = 1 and k = 2 ls
// orders them (above every k below), a box without volume (-inf) included.
__device__ __forceinline__ void finish_subvolume(const MergeArgs &a, int64_t s, double m) {
    const int lane = threadIdx.x & 31, R = a.R, K = sum_count(R);
    double *slot = a.slots + s * (K + 3);
    const double n = static_cast<double>(a.samples[s]);
    // One logarithm a lane: of the product of its widths, kept in [1, 2) by its exponent, and, on the first lane
    // without a width (the next round's first lane if all have one), of n.  A width that is no positive normal
    // number sends the warp to a logarithm per width.
    double log_vol = 0.0, p = 1.0;
    long long e = 0;
    bool plain = true;
    for (int j = lane; j < a.d; j += 32) {
        const double x = p * (a.hi[s * a.d + j] - a.lo[s * a.d + j]);
        const int hi32 = __double2hiint(x), ex = (hi32 >> 20) & 0x7ff;
        plain = plain && hi32 > 0 && ex != 0 && ex != 0x7ff;
        e += ex - 1023;
        p = __hiloint2double((hi32 & 0x000fffff) | 0x3ff00000, __double2loint(x));
    }
    const int n_lane = a.d & 31;
    const bool spare = a.d < 32;
    log_vol = log(spare && lane == n_lane ? n : p);
    double log_n = __shfl_sync(0xffffffffu, log_vol, n_lane);
    if (!spare) log_n = log(n);
    else if (lane == n_lane) log_vol = 0.0;
    if (__all_sync(0xffffffffu, plain)) {
        log_vol = fma(static_cast<double>(e), 0.69314718055994531, log_vol);
    } else {
        log_vol = 0.0;
        for (int j = lane; j < a.d; j += 32) log_vol += log(a.hi[s * a.d + j] - a.lo[s * a.d + j]);
    }
    log_vol = a.log_norm_set ? a.log_norm : warp_sum_f64(log_vol);
    if (lane == 0) {
        slot[0] = n;
        slot[1] = m;
        slot[2] = log_vol;
    }
    __syncwarp();
    const double sw = slot[3], sw2 = slot[4];
    double tt = 0.0, gt = 0.0, k = 0.0;
    if (n > 0.0 && sw > 0.0) {
        const double ls = log_vol - log_n - m;
        k = 2.0 * ls;
        tt = 1.0;
        if ((__double2hiint(ls) & 0x7fffffff) < kFarLog) {
            // ln 2 in two parts, the upper one of 32 bits (Cody & Waite's reduction)
            k = rint(ls * 1.4426950408889634);
            tt = exp(fma(-k, 1.9082149292705877e-10, fma(-k, 0.69314718036912382, ls)));
        }
        if (n >= 2.0) gt = tt * tt / (n - 1.0);
    }
    const int64_t c0 = a.chunk_off[s];
    double *q = a.partials + c0 * (K + 2);
    const bool room = a.chunk_off[s + 1] > c0;  // else n = 0 and nothing of it is read
    if (lane == 0) {
        a.f_buf[s] = tt;
        a.f_buf[a.nsub + s] = gt;
        if (room) {
            q[0] = k;
            q[1] = n * sw2 - sw * sw;
        }
    }
    for (int r = lane; r < R; r += 32) {
        const double s1 = slot[5 + r] * a.inv_d, s2 = slot[5 + R + r] * a.inv_d,
                     s3 = slot[5 + 2 * R + r] * (a.inv_d * a.inv_d);
        slot[5 + r] = s1;
        slot[5 + R + r] = s2;
        slot[5 + 2 * R + r] = s3;
        if (room) {
            q[2 + r] = n * s3 - s1 * s1;
            q[2 + R + r] = n * s2 - sw * s1;
        }
    }
}

// Cross-subvolume merge by one CTA, every order fixed by nsub and R:
//   Z' = sum f_s sum w,  N'(r) = sum f_s sum w P_r,  C = N'/Z'
//   Var Z' = sum g_s V_Z,  Var C = sum g_s [V_N - 2 C Cov + C^2 V_Z] / Z'^2
// (delta method; g_s = f_s^2 / (n_s - 1)).  For the sums over s of R terms
// each, a warp takes 32 / rp subvolumes at a time, rp >= R lanes for each.
__device__ void merge_slots(const MergeArgs &a) {
    __shared__ double sh[5][kMergeWarps], part[kMergeWarps][32], s_all[5], s_c[32];
    __shared__ long long s_key;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int R = a.R, K = sum_count(R), SL = K + 3;
    const int64_t nsub = a.nsub;
    auto record = [&](int64_t s) { return a.partials + a.chunk_off[s] * (K + 2); };
    if (tid == 0) s_key = LLONG_MIN;
    __syncthreads();
    long long key = LLONG_MIN;
    for (int64_t s = tid; s < nsub; s += kMergeThreads)
        if (!is_zero(__ldcg(a.f_buf + s))) key = max(key, order_f64(__ldcg(record(s))));
    if (key != LLONG_MIN) atomicMax(&s_key, key);
    __syncthreads();
    key = s_key;  // LLONG_MIN: no subvolume has weight
    const double kmax = unorder_f64(key);
    double z = 0.0, vz = 0.0;
    unsigned long long n_tot = 0;
    int used = 0, bad = 0;
    for (int64_t s = tid; s < nsub; s += kMergeThreads) {
        const uint64_t n = a.samples[s];
        double f = __ldcg(a.f_buf + s), g = __ldcg(a.f_buf + nsub + s);
        n_tot += n;
        used += n > 0;
        if (!is_zero(f)) {
            const double *q = record(s);
            const double k = __ldcg(q) - kmax;
            if (k >= -1100.0) {
                f *= pow2(static_cast<int>(k));
                g *= pow2(2 * static_cast<int>(k));
            } else {
                f = g = k < 0.0 ? 0.0 : NAN;  // no finite kmax, or an ls that is no number
            }
            z = fma(f, __ldcg(a.slots + s * SL + 3), z);
            if (n < 2) bad = 1;
            else vz = fma(g, __ldcg(q + 1), vz);
        }
        a.f_buf[s] = f;
        a.f_buf[nsub + s] = g;  // 0 for n < 2
    }
    if (warp * 32 < nsub) {
        z = warp_sum_f64(z);
        vz = warp_sum_f64(vz);
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) n_tot += __shfl_xor_sync(0xffffffffu, n_tot, off);
        used = __reduce_add_sync(0xffffffffu, used);
        bad = __reduce_or_sync(0xffffffffu, bad);
    }
    if (lane == 0) {
        sh[0][warp] = z;
        sh[1][warp] = vz;
        sh[2][warp] = static_cast<double>(n_tot);
        sh[3][warp] = used;
        sh[4][warp] = bad;
    }
    __syncthreads();
    if (tid < 5) {
        double v = 0.0;
        for (int w = 0; w < kMergeWarps && w * 32 < nsub; ++w) v += sh[tid][w];
        s_all[tid] = v;
    }
    __syncthreads();
    const bool inf_err = s_all[4] > 0.0;
    // sum over s of term(s), s in the order (warp, lane group), then lane groups, then warps: in lanes r of warp 0
    auto sum = [&](int rn, int rp, auto term) {
        const int r = lane & (rp - 1), groups = 32 / rp, step = kMergeWarps * groups;
        const bool mine = r < rn;
        double v = 0.0;
#pragma unroll 4
        for (int64_t s = warp * groups + lane / rp; s < nsub; s += step)
            if (mine) v = term(s, r, v);
        if (warp * groups < nsub)
            for (int off = rp; off < 32; off *= 2) v += __shfl_xor_sync(0xffffffffu, v, off);
        __syncthreads();
        if (lane < rn) part[warp][lane] = v;
        __syncthreads();
        double total = 0.0;
        if (warp == 0 && lane < rn)
            for (int w = 0; w < kMergeWarps && w * groups < nsub; ++w) total += part[w][lane];
        return total;
    };
    if (warp == 1 && lane < 2) {  // beside the products' sums of the other warps
        const double Z = s_all[0];
        if (lane == 0)
            a.totals[0] = key == LLONG_MIN ? -INFINITY
                                              : fma(kmax, fabs(kmax) < 0x1p61 ? 0.69314718055994531 : 0.5, log(Z));
        else
            a.totals[1] = inf_err ? INFINITY : sqrt(s_all[1] > 0.0 ? s_all[1] : 0.0) / Z;
        a.totals[2 + lane] = s_all[2 + lane];
    }
    for (int r0 = 0; r0 < R; r0 += 32) {
        const int rn = min(32, R - r0);
        int rp = 1;
        while (rp < rn) rp *= 2;
        const double N = sum(rn, rp, [&](int64_t s, int r, double v) {
            return fma(a.f_buf[s], __ldcg(a.slots + s * SL + 5 + r0 + r), v);
        });
        if (warp == 0 && lane < rn) s_c[lane] = N / s_all[0];
        __syncthreads();
        const double C = s_c[(lane & (rp - 1)) < rn ? lane & (rp - 1) : 0], C2 = C * C, m2C = -2.0 * C;
        const double V = sum(rn, rp, [&](int64_t s, int r, double v) {
            const double g = a.f_buf[nsub + s];
            if (is_zero(g)) return v;
            const double *q = record(s);
            const double var = fma(C2, __ldcg(q + 1), fma(m2C, __ldcg(q + 2 + R + r0 + r), __ldcg(q + 2 + r0 + r)));
            return fma(g, var, v);
        });
        if (warp == 0 && lane < rn) {
            a.totals[4 + r0 + lane] = C;
            a.totals[4 + R + r0 + lane] = inf_err ? INFINITY : sqrt(V > 0.0 ? V : 0.0) / s_all[0];
        }
    }
}

// The first 'active' warps of every CTA take a task each, CTA by CTA: tasks
// 0 .. nsub - 1 are the subvolumes; where subvolumes have more than
// kMergeWhole chunks, the next a.windows tasks are the windows of kMergePiece
// chunks [32 j, 32 j + 32): the one subvolume that began before the window
// owns a piece of it, whose merged record replaces the piece's first chunk
// record.  The CTA that arrives last (a counter, zeroed per execution) merges
// those pieces and then all slots.  A subvolume's pieces follow from the chunk
// table, so every order is fixed by the job.  80 registers: left alone it takes
// 102, and its CTAs start later beside a batch's other kernels (32 jobs 39.52
// -> 39.42 ms; 64 spill, one volume of 1024 chunks 71.5 -> 73.6 us a pass).
__global__ void __maxnreg__(80) merge_records(const MergeArgs a, int active) {
    __shared__ bool s_last;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int R = a.R, K = sum_count(R);
    auto merge = [&](double *out, int64_t count, auto at) {
        return merge_list(count, R, at, [&](int k, double v) { out[k] = v; });
    };
    auto piece = [&](int64_t c0, int64_t c1) {  // merged record of chunks [c0, c1) in place of the first
        double *q = a.partials + c0 * (K + 2);
        const double m = merge(q + 2, c1 - c0, [&](int64_t i) { return a.partials + (c0 + i) * (K + 2); });
        __syncwarp();
        if (lane == 0) q[1] = m;
    };
    const int64_t task = warp < active ? blockIdx.x * static_cast<int64_t>(active) + warp : a.nsub + a.windows;
    if (task < a.nsub) {
        const int64_t c0 = a.chunk_off[task], c1 = a.chunk_off[task + 1];
        if (c1 - c0 <= kMergeWhole) {
            const double m = merge(a.slots + task * (K + 3) + 3, c1 - c0,
                                   [&](int64_t i) { return a.partials + (c0 + i) * (K + 2); });
            finish_subvolume(a, task, m);
        } else {
            piece(c0, (c0 / kMergePiece + 1) * kMergePiece);
        }
    } else if (task < a.nsub + a.windows) {
        const int64_t c = (task - a.nsub) * kMergePiece;
        if (c < a.chunk_off[a.nsub]) {
            const int64_t s = find_subvolume(a.chunk_off, a.nsub, c), c0 = a.chunk_off[s], c1 = a.chunk_off[s + 1];
            if (c1 - c0 > kMergeWhole && c0 < c) piece(c, min(c1, c + kMergePiece));
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        s_last = atomicAdd(a.arrived, 1ull) + 1ull == gridDim.x;
        __threadfence();
    }
    __syncthreads();
    if (!s_last) return;
    if (a.windows > 0) {
        for (int64_t s = warp; s < a.nsub; s += kMergeWarps) {
            const int64_t c0 = a.chunk_off[s], c1 = a.chunk_off[s + 1];
            if (c1 - c0 <= kMergeWhole) continue;
            // the pieces' records lie at c0 and at every multiple of kMergePiece in (c0, c1)
            const int64_t w0 = c0 / kMergePiece, pieces = (c1 - 1) / kMergePiece - w0 + 1;
            const double m = merge(a.slots + s * (K + 3) + 3, pieces, [&](int64_t i) {
                return a.partials + (i == 0 ? c0 : (w0 + i) * kMergePiece) * (K + 2);
            });
            finish_subvolume(a, s, m);
        }
        __syncthreads();
    }
    merge_slots(a);
}

// ---------------------------------------------------------------------------
// Single-step kernels for step-by-step checks.
// ---------------------------------------------------------------------------
template <typename Real>
__global__ void points_kernel(const PointsArgs a, const RoundKeys rk) {
    const int64_t idx = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
    const int nq = (a.d + 3) / 4;
    if (idx >= a.count * nq) return;
    const int64_t k = idx / nq;
    const int q = static_cast<int>(idx % nq);
    const uint64_t i = a.first + static_cast<uint64_t>(k);
    const uint4 wd = philox4x32_10(
        make_uint4(static_cast<uint32_t>(q), static_cast<uint32_t>(i), static_cast<uint32_t>(i >> 32), a.sub_id), rk);
    const uint32_t w4[4] = {wd.x, wd.y, wd.z, wd.w};
    for (int t = 0; t < 4; ++t) {
        const int j = 4 * q + t;
        if (j >= a.d) break;
        Real b, w;
        BoxPair<Real>::load(a.lo, a.hi, j, b, w);
        a.y[k * a.d + j] = static_cast<double>(Coord<Real>::map(w4[t], b, w));
    }
}

const ShapeKernels *find_shape(int nx, int nt) {
    for (auto table : {shapes_small, shapes_config_a, shapes_config_b, shapes_config_c, shapes_config_d}) {
        int n = 0;
        const ShapeKernels *t = table(&n);
        for (int i = 0; i < n; ++i)
            if (t[i].nx == nx && t[i].nt == nt) return &t[i];
    }
    return generic_shape(nx, nt);
}

cudaError_t launch_merges(const MergeArgs &m, cudaStream_t st) {
    // as few of a CTA's warps as keep the grid near one CTA per SM: they share the SM's FP64 pipe
    const int64_t tasks = m.nsub + m.windows;
    const int64_t active = std::min<int64_t>(kMergeWarps, (tasks + kMergeSpread - 1) / kMergeSpread);
    const int64_t blocks = (tasks + active - 1) / active;
    merge_records<<<static_cast<unsigned>(blocks), kMergeThreads, 0, st>>>(m, static_cast<int>(active));
    return cudaGetLastError();
}

cudaError_t launch_points(const PointsArgs &a, bool fp32, uint32_t seed, uint32_t job, cudaStream_t st) {
    const int threads = 128;
    const int64_t work = a.count * ((a.d + 3) / 4);
    const int64_t blocks = (work + threads - 1) / threads;
    if (blocks == 0) return cudaSuccess;
    if (fp32)
        points_kernel<float><<<static_cast<unsigned>(blocks), threads, 0, st>>>(a, make_round_keys(seed, job));
    else
        points_kernel<double><<<static_cast<unsigned>(blocks), threads, 0, st>>>(a, make_round_keys(seed, job));
    return cudaGetLastError();
}

}  // namespace bfi
