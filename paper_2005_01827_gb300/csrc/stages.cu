// stages.cu -- data-preparation and template kernels of the batched LISA likelihood (Katz et al. 2020, Sec. II.A).
#include "kernels.h"
#include "model.cuh"

namespace lisa {

// f_j = f0 + j df, rounded as a separate product and sum (no fused multiply-add) so
// that band edges and knot-to-bin boundaries are decided exactly as written.
__device__ __forceinline__ double bin_freq(double f0, double df, int j) {
    return __dadd_rn(f0, __dmul_rn((double)j, df));
}

// ---------------------------------------------------------------------------- data prep
// w = 4 df / S and w d per bin and channel (Eq. (3)), the partial sums of <d|d>, and a
// flag for a non-positive or non-finite PSD value or a non-finite data value.
__global__ void __launch_bounds__(256) prep_kernel(const double *d, const double *psd, int N,
                                                   double df, double *bins, double *ddpart,
                                                   int *bad) {
    __shared__ double red[8];
    double acc = 0.0;
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < N; j += gridDim.x * blockDim.x) {
        double *o = bins + (size_t)j * kBinDoubles;
        for (int c = 0; c < 3; c++) {
            const double S = psd[(size_t)c * N + j];
            const double dr = d ? d[2 * ((size_t)c * N + j)] : 0.0;
            const double di = d ? d[2 * ((size_t)c * N + j) + 1] : 0.0;
            if (!(S > 0.0) || !isfinite(S) || !isfinite(dr) || !isfinite(di)) atomicExch(bad, 1);
            const double wgt = 4.0 * df / S;
            o[c] = wgt;
            o[3 + 2 * c] = wgt * dr;
            o[4 + 2 * c] = wgt * di;
            acc += wgt * (dr * dr + di * di);
        }
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int i = 0; i < (int)(blockDim.x >> 5); i++) t += red[i];
        ddpart[blockIdx.x] = t;
    }
}

int prep_blocks(int N) {
    const int b = (N + 255) / 256;
    return b < kPrepBlocks ? b : kPrepBlocks;
}

cudaError_t launch_prep(const double *d, const double *psd, int N, double df, double *bins,
                        double *ddpart, int *bad, cudaStream_t s) {
    prep_kernel<<<prep_blocks(N), 256, 0, s>>>(d, psd, N, df, bins, ddpart, bad);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------- template
// Materialise the dense template of walker 0 (injections and element-wise checks):
// one thread per bin, the same segment rule and evaluation as the fused kernel.
__device__ __forceinline__ int find_segment(const int *kb, int K, int j) {
    int lo = 0, hi = K - 2;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (kb[mid] <= j)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

__global__ void __launch_bounds__(256) template_kernel(StageDims d, StageBufs b, double *out) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= d.N) return;
    const double f = bin_freq(d.f0, d.df, j);
    double h[6] = {0, 0, 0, 0, 0, 0};
    if (b.valid[0]) {
        const double wt = kTwoPi * b.tc[0];
        for (int mi = 0; mi < d.L; mi++) {
            const int *bd = b.band + (size_t)mi * 3;
            if (!bd[0] || j < bd[1] || j > bd[2]) continue;
            const int s = find_segment(b.kb + (size_t)mi * d.K, d.K, j);
            const double x = f - b.fk[(size_t)mi * d.K + s];
            const double *c = b.coef + ((size_t)mi * (d.K - 1) + s) * 32;
            double v[kNSeries];
            for (int q = 0; q < kNSeries; q++)
                v[q] = c[4 * q] + x * (c[4 * q + 1] + x * (c[4 * q + 2] + x * c[4 * q + 3]));
            double sn, cs;
            sincos(fma(-wt, f, v[1]), &sn, &cs);
            const double zr = v[0] * cs, zi = v[0] * sn;
            for (int ch = 0; ch < 3; ch++) {
                const double tr = v[2 + 2 * ch], ti = v[3 + 2 * ch];
                h[2 * ch] += tr * zr - ti * zi;
                h[2 * ch + 1] += tr * zi + ti * zr;
            }
        }
    }
    for (int ch = 0; ch < 3; ch++) {
        out[2 * ((size_t)ch * d.N + j)] = h[2 * ch];
        out[2 * ((size_t)ch * d.N + j) + 1] = h[2 * ch + 1];
    }
}

cudaError_t launch_template(const StageDims &d, const StageBufs &b, double *out, cudaStream_t s) {
    template_kernel<<<(d.N + 255) / 256, 256, 0, s>>>(d, b, out);
    return cudaGetLastError();
}

}  // namespace lisa
