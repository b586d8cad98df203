// spline.cu -- not-a-knot cubic splines of the knot values (the Scipy-type tridiagonal
// solve of Katz et al. 2020, Sec. II.A) and the FP64 cubic coefficients.
//
// One block per (walker, mode) system; the unknowns are the second derivatives
// M_1 .. M_{K-2} of each of the 8 series, not-a-knot eliminating M_0 and M_{K-1}.  The
// matrix (shared by the series) has diagonal 2 (h_{i-1} + h_i) and off-diagonals h_{i-1},
// h_i, so whatever a sweep starts from is forgotten by a factor of 1 / (1 + r + sqrt(1 + r + r^2))
// a row for a step ratio r: 0.27 on the nearly even steps of many log-spaced knots.  So every
// thread sweeps a chunk of rows of its own after a run-in of halo rows, and a sweep of 1022 rows
// takes 64 steps instead of 1022.  The rows of the run-in grow towards low frequencies, M of the
// phase as f^(-11/3), r^(11/3) a row: of the row's own value the run-in's start is left with
// (r^(11/3) / (1 + r + sqrt(1 + r + r^2)))^halo.  With few knots over several decades that falls slowly
// (40 knots over five: 0.7 a row), so the run-in follows from r: 32 rows for 128 knots over two decades
// or 1024 over any, 37 for 128 and 51 for 64 knots over five decades (with 32 throughout 40
// knots were off by 6e-9 of the row's own value over four decades, 3e-11 rad of a phase of 1e5 rad, and by 2e-6
// over five).  The pivots forget by r / (1 + r + sqrt(1 + r + r^2))^2, 0.07, a row and do not
// grow: 16 rows.
//
// What bounds it: with few systems the latency of the sweep steps, so the series are dealt
// to several blocks; with many systems the FP64 pipe (2 lanes per clock per SM): slopes and
// right-hand sides and the divisions by the pivots are independent and use full warps, a sweep
// step is one FP64 operation (the quotients are formed first, and pivots come as ratios of
// minors, so that no division is in a chain: with divisions in the chain 39 us, 82 us, 3.11 and
// 1.57 ms for the cases below).  Measured on GB300 (solve and coefficient kernel) against one
// system per lane of one warp with every row in series: 1 system of 256 knots 367 -> 31 us,
// 148 systems of 509 knots 938 -> 58 us, 6144 systems of 1024 knots 3.66 -> 2.71 ms in FP64
// and 2.29 -> 1.45 ms in split precision.
#include "kernels.h"
#include "model.cuh"

namespace lisa {

namespace {
constexpr int kThreads = 256;
// run-in rows of a sweep of n rows at the step ratio r = x1 / x0 of its knots: until less than 2^-53 of
// a row's own value is left of what it started from
__device__ __forceinline__ int sweep_halo(double x0, double x1, int n) {
    const float r = (float)x1 / (float)x0;
    const float lost = log2f(1.0f + r + sqrtf(fmaf(r, r, 1.0f + r))) - 11.0f / 3.0f * log2f(r);  // bits a row
    const float rows = 54.0f / lost;
    return lost > 0.0f && rows < (float)n ? max(32, (int)rows + 1) : n;
}
constexpr int kPivotHalo = 16;   // run-in rows of the pivots
constexpr size_t kMaxSmem = 227 * 1024;
}  // namespace

// Row arrays in shared memory hold entry i at at(i): chunks of C = 2^cs entries with an odd
// pitch, so that threads sweeping different chunks hit different banks.
struct Rows {
    int cs, mask, pitch;
    __host__ __device__ __forceinline__ int at(int i) const { return (i >> cs) * pitch + (i & mask); }
};

// chunk layout for `tps` sweeping threads per series
__host__ __device__ inline Rows rows_of(int K, int tps) {
    Rows r;
    r.cs = 0;
    while ((tps << r.cs) < K - 1) r.cs++;
    r.mask = (1 << r.cs) - 1;
    r.pitch = r.cs ? (1 << r.cs) + 1 : 1;
    return r;
}

// Sweeping threads per series of a block that owns nq series.  A step has a latency of about
// 50 clocks and takes 32 of the pipe per warp, so few warps with longer chunks (less run-in) are
// best: the solve of one system of 256 (1024) knots, one series a block, 256 threads 25.6 (46.4)
// us, 128 24.4 (44.3), 64 24.6 (44.8), 32 24.8 (46.7).
__host__ __device__ inline int sweep_threads(int nq) { return nq > 1 ? 32 : 64; }

// Forward sweep of one chunk: rp_i = rhs_i / pivot_i - (sub_i / pivot_i) rp_{i-1} in place, the
// quotients in y and sd.  `store` selects the chunk itself (the run-in stores nothing).
template <typename T>
__device__ __forceinline__ T sweep_forward(T *y, const T *sd, const Rows R, int from, int to, T prev,
                                           bool store) {
    for (int i = from; i < to; i++) {
        const int o = R.at(i);
        prev = y[o] - sd[o] * prev;
        if (store) y[o] = prev;
    }
    return prev;
}

// Backward sweep of one chunk: M_i = rp_i - c_i M_{i+1}, rows to-1 down to from.
template <typename T>
__device__ __forceinline__ T sweep_backward(T *y, const T *c, const Rows R, int from, int to, int n,
                                            T next, bool store) {
    for (int i = to - 1; i >= from; i--) {
        const int o = R.at(i);
        next = (i == n - 2) ? y[o] : y[o] - c[o] * next;
        if (store) y[o] = next;
    }
    return next;
}

// One stage of a series' solve (a barrier follows each): run-in and chunk of the forward
// sweep, run-in and chunk of the backward sweep, the not-a-knot ends.  The run-ins read
// entries that the neighbours' chunks overwrite, hence stages of their own.
template <typename T>
__device__ __forceinline__ void solve_stage(int stage, T &v, T *y, const T *h, const T *ih,
                                            const T *sd, const T *c, const Rows R, int t, int n, int halo) {
    const int C = R.mask + 1;
    const int i0 = 1 + t * C, i1 = min(i0 + C, n - 1);
    if (stage == 4) {  // M_0 and M_{K-1} from their neighbours
        if (t != 0) return;
        const T h0 = h[R.at(0)], h1 = h[R.at(1)], ha = h[R.at(n - 3)], hb = h[R.at(n - 2)];
        y[R.at(0)] = ((h0 + h1) * y[R.at(1)] - h0 * y[R.at(2)]) * ih[R.at(1)];
        y[R.at(n - 1)] = ((ha + hb) * y[R.at(n - 2)] - hb * y[R.at(n - 3)]) * ih[R.at(n - 3)];
        return;
    }
    if (i0 >= n - 1) return;
    if (stage == 0) v = sweep_forward(y, sd, R, max(1, i0 - halo), i0, T(0), false);
    if (stage == 1) sweep_forward(y, sd, R, i0, i1, v, true);
    if (stage == 2) v = sweep_backward(y, c, R, i1, min(n - 1, i1 + halo), n, T(0), false);
    if (stage == 3) sweep_backward(y, c, R, i0, i1, n, v, true);
}

// kSplit: the phase (series 1) in FP64, the other seven in FP32 from their FP32 knot values
// (the interpolant depends on M only through terms of order h^2 M, far below the values).
// Block (s, y) owns series [y, y + 1) 8 / gridDim.y of system s.
template <bool kSplit>
__global__ void __launch_bounds__(kThreads) spline_kernel(StageDims d, StageBufs b) {
    extern __shared__ __align__(16) unsigned char spl_sm[];
    const int K = d.K, n = K, tid = threadIdx.x;
    const size_t wm = blockIdx.x;
    if (!b.band[wm * 3]) return;  // inactive modes (and invalid walkers) have no splines
    const int per = kNSeries / gridDim.y;
    const int q0 = blockIdx.y * per;
    const int tps = sweep_threads(per);
    const Rows R = rows_of(K, tps);
    const int NP = R.at(K - 1) + 1;
    double *h = reinterpret_cast<double *>(spl_sm), *ih = h + NP, *sd = ih + NP, *c = sd + NP;
    // FP64 series, then (split) the FP32 copies of the matrix and the FP32 series; a block of
    // one series holds only the kind it owns
    double *ys = c + NP;  // [1 or per][NP]
    float *h32 = reinterpret_cast<float *>(ys + (!kSplit ? per : per == 1 && q0 != 1 ? 0 : 1) * NP);
    float *ih32 = h32 + NP, *sd32 = ih32 + NP, *c32 = sd32 + NP;
    float *ys32 = c32 + NP;  // split: [per][NP] (phase slot unused)
    const bool own32 = kSplit && !(per == 1 && q0 == 1);
    const double *x = b.fk + wm * K;
    const int halo = sweep_halo(x[0], x[1], n);
    const double *yg = b.vals + wm * kNSeries * (size_t)K;
    const float *y32g = split_vals32(b.vals, wm, K);

    for (int i = tid; i < n - 1; i += kThreads) {
        const double hi = x[i + 1] - x[i], v = 1.0 / hi;
        const int o = R.at(i);
        h[o] = hi;
        ih[o] = v;
        if (own32) {
            h32[o] = (float)hi;
            ih32[o] = (float)v;
        }
    }
    __syncthreads();
    // Warp 0: pivots of its chunk of rows, as ratios p_i / p_{i-1} of the leading minors p_i =
    // dia_i p_{i-1} - sub_i sup_{i-1} p_{i-2} (in units of the chunk's first step), which have no
    // division in the chain; left as p_i in c and p_{i-1} in sd.  The other warps: right-hand
    // sides 6 (slope_i - slope_{i-1}) of the block's series
    if (tid < 32) {
        const int F = (n - 2 + 31) / 32, i0 = 1 + tid * F, i1 = min(i0 + F, n - 1);
        const int is = max(1, i0 - kPivotHalo);
        const double unit = is < n - 1 ? ih[R.at(is)] : 0.0;
        double pm = 0.0, p = 1.0, sup = 0.0;  // p_{i-2}, p_{i-1}, sup_{i-1}
        for (int i = is; i < i1; i++) {
            const int o = R.at(i), om = R.at(i - 1);
            const double hp = h[om], hc = h[o];
            double dia = 2.0 * (hp + hc), sb = hp, su = hc;
            if (i == 1) {
                dia += hp * (hp + hc) * ih[o];
                su -= hp * hp * ih[o];
            }
            if (i == n - 2) {
                dia += hc * (hp + hc) * ih[om];
                sb -= hc * hc * ih[om];
            }
            const double w = (sb * unit) * (sup * unit) * pm;
            pm = p;
            p = fma(dia * unit, p, -w);
            sup = su;
            if (i >= i0) {
                sd[o] = pm * unit;
                c[o] = p;
            }
        }
    } else {
        for (int q = q0; q < q0 + per; q++) {
            if (kSplit && q != 1) {
                const float *y = y32g + (size_t)(q == 0 ? 0 : q - 1) * K;
                float *o32 = ys32 + (size_t)(q - q0) * NP;
                for (int i = 1 + tid - 32; i < n - 1; i += kThreads - 32) {
                    const float sl = (y[i + 1] - y[i]) * ih32[R.at(i)];
                    const float sp = (y[i] - y[i - 1]) * ih32[R.at(i - 1)];
                    o32[R.at(i)] = 6.0f * (sl - sp);
                }
            } else {
                const double *y = yg + (size_t)q * K;
                double *o64 = ys + (size_t)(kSplit ? 0 : q - q0) * NP;
                for (int i = 1 + tid - 32; i < n - 1; i += kThreads - 32) {
                    const double sl = (y[i + 1] - y[i]) * ih[R.at(i)];
                    const double sp = (y[i] - y[i - 1]) * ih[R.at(i - 1)];
                    o64[R.at(i)] = 6.0 * (sl - sp);
                }
            }
        }
    }
    __syncthreads();
    // divide by the pivots: sub- and super-diagonal, right-hand sides
    for (int i = 1 + tid; i < n - 1; i += kThreads) {
        const int o = R.at(i), om = R.at(i - 1);
        const double hp = h[om], hc = h[o], v = sd[o] / c[o];
        const double s = (i == 1) ? 0.0 : (i == n - 2) ? hp - hc * hc * ih[om] : hp;
        const double u = (i == 1) ? hc - hp * hp * ih[o] : hc;
        sd[o] = s * v;
        c[o] = u * v;
        if (own32) {
            sd32[o] = (float)(s * v);
            c32[o] = (float)(u * v);
        }
        for (int q = q0; q < q0 + per; q++) {
            if (kSplit && q != 1)
                ys32[(size_t)(q - q0) * NP + o] *= (float)v;
            else
                ys[(size_t)(kSplit ? 0 : q - q0) * NP + o] *= v;
        }
    }
    __syncthreads();
    // a series' threads lie in whole warps, so the FP64 / FP32 choice is uniform per warp
    const int ql = tid / tps, t = tid % tps;
    double v64 = 0.0;
    float v32 = 0.0f;
    for (int stage = 0; stage < 5; stage++) {
        if (ql < per) {
            if (kSplit && q0 + ql != 1)
                solve_stage<float>(stage, v32, ys32 + (size_t)ql * NP, h32, ih32, sd32, c32, R, t, n, halo);
            else
                solve_stage<double>(stage, v64, ys + (size_t)(kSplit ? 0 : ql) * NP, h, ih, sd, c, R, t, n, halo);
        }
        __syncthreads();
    }

    // second derivatives, 1/h and (split) the FP32 copies, coalesced
    double *Mg = b.mscratch + wm * kScratchRows * (size_t)K;
    float *M32g = split_m32(b.mscratch, wm, K), *F32g = split_fac32(b.mscratch, wm, K);
    for (int q = q0; q < q0 + per; q++) {
        if (kSplit && q != 1) {
            const float *y = ys32 + (size_t)(q - q0) * NP;
            float *o = M32g + (size_t)(q == 0 ? 0 : q - 1) * K;
            for (int i = tid; i < n; i += kThreads) o[i] = y[R.at(i)];
        } else {
            const double *y = ys + (size_t)(kSplit ? 0 : q - q0) * NP;
            for (int i = tid; i < n; i += kThreads) Mg[(size_t)q * K + i] = y[R.at(i)];
        }
    }
    if (q0 == 0) {
        for (int i = tid; i < n - 1; i += kThreads) {
            Mg[kNSeries * (size_t)K + i] = ih[R.at(i)];
            if (kSplit) {
                F32g[i] = ih32[R.at(i)];
                F32g[K + i] = h32[R.at(i)];
            }
        }
    }
}

// Cubic coefficients of every (system, segment, series) from the second derivatives, as
// a grid-stride kernel of its own (full occupancy whatever the solve's blocks hold).
// kSplit: only the FP64 phase series (the others stay as FP32 values and second
// derivatives for the segment records).
template <bool kSplit>
__global__ void __launch_bounds__(256) spline_coef_kernel(StageDims d, StageBufs b) {
    const int K = d.K;
    const long long per_sys = (long long)(K - 1) * (kSplit ? 1 : kNSeries);
    const long long total = (long long)d.B * d.L * per_sys;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
         t += (long long)gridDim.x * blockDim.x) {
        const long long w2 = t / per_sys;
        const int rem = (int)(t - w2 * per_sys);
        if (!b.band[w2 * 3]) continue;
        const int sgm = kSplit ? rem : rem / kNSeries, q = kSplit ? 1 : rem % kNSeries;
        const double *x2 = b.fk + (size_t)w2 * K;
        const double *M2 = b.mscratch + (size_t)w2 * kScratchRows * K;
        const double *yq = b.vals + ((size_t)w2 * kNSeries + q) * K;
        const double *Mq = M2 + (size_t)q * K;
        const double h = x2[sgm + 1] - x2[sgm], hi = M2[(size_t)kNSeries * K + sgm];
        const double m0 = Mq[sgm], m1 = Mq[sgm + 1];
        double *c = b.coef + ((size_t)w2 * (K - 1) + sgm) * 32 + q * 4;
        c[0] = yq[sgm];
        c[1] = (yq[sgm + 1] - yq[sgm]) * hi - h * (2.0 * m0 + m1) * (1.0 / 6.0);
        c[2] = 0.5 * m0;
        c[3] = (m1 - m0) * hi * (1.0 / 6.0);
    }
}

namespace {

template <bool kSplit>
size_t spline_smem(int K, int per) {
    const Rows R = rows_of(K, sweep_threads(per));
    const size_t NP = R.at(K - 1) + 1;
    if (!kSplit) return NP * 8 * (4 + per);
    return per == 1 ? NP * (8 * 4 + 4 * 5) : NP * (8 * 5 + 4 * (4 + per));
}

// Blocks per system: one while the systems fill the chip's 152 SMs, more (each with fewer
// series, the pivots repeated) while they do not or while a block's rows would not fit in
// shared memory (K above about 2300).  Solve and coefficients with 1, 2, 4, 8 blocks a system: one
// system of 256 knots 35, 33, 31, 31 us, 148 systems of 509 knots 58, 62, 70, 105 us.
template <bool kSplit>
int spline_blocks(int nsys, int K) {
    int y = 1;
    while (y < kNSeries && nsys * y * 2 <= 152) y *= 2;
    while (y < kNSeries && spline_smem<kSplit>(K, kNSeries / y) > kMaxSmem) y *= 2;
    return y;
}

template <bool kSplit>
cudaError_t launch_spline_t(const StageDims &d, const StageBufs &b, cudaStream_t s) {
    const int nsys = d.B * d.L, y = spline_blocks<kSplit>(nsys, d.K);
    const size_t smem = spline_smem<kSplit>(d.K, kNSeries / y);
    cudaError_t e = cudaFuncSetAttribute(spline_kernel<kSplit>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    spline_kernel<kSplit><<<dim3(nsys, y), kThreads, smem, s>>>(d, b);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const long long total = (long long)nsys * (d.K - 1) * (kSplit ? 1 : kNSeries);
    const long long want = (total + 255) / 256, cap = 152LL * 8;  // 8 blocks per SM
    const int blocks = (int)(want < cap ? want : cap);
    spline_coef_kernel<kSplit><<<blocks, 256, 0, s>>>(d, b);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_spline(const StageDims &d, const StageBufs &b, cudaStream_t s) {
    return launch_spline_t<false>(d, b, s);
}

cudaError_t launch_spline_split(const StageDims &d, const StageBufs &b, cudaStream_t s) {
    return launch_spline_t<true>(d, b, s);
}

}  // namespace lisa
