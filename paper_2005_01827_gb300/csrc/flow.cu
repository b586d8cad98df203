// flow.cu -- the normalizing-flow proposal of include/lisa_flow.h: evaluation in both
// directions, training (forward, back-propagation, Adam) and the independence
// Metropolis-Hastings step of the sampler (Eq. (13)).
//
// Every network layer is a GEMM on the tensor cores: bfloat16 operands, FP32 accumulation,
// mma.sync.m16n8k16.  The networks are small (128 x 128) and the batches few hundred to a few
// thousand samples, so what bounds a pass is the latency of its 24 layers one after another,
// not arithmetic.  Hence the smallest unit the instruction has: a block holds 16 samples, its
// eight warps share a layer's outputs (16 columns each), and as each weight is then used by
// one warp only, it goes from L2 to that warp's registers in the order of the instruction's
// fragments (packed so by the optimiser), fetched for the next coupling as soon as this one's are
// used; no staging of weights in shared memory, four block barriers a coupling.  256 samples in
// both directions, two calls: 156 -> 37 us (64 samples a block, weights staged between barriers).
//
// Training keeps a coupling's activations in shared memory for the backward pass and writes
// the operands of the weight gradients, contractions over the samples, to global memory in
// fragment order; a second kernel reduces them without atomics, 16 x 128 weights a block, and
// goes on to the Adam step and the packed copies of the weights it owns.  One iteration, 1024
// samples: 840 -> 53 us.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <string>
#include <vector>

#include "../../include/lisa_flow.h"
#include "flow.h"
#include "internal.h"
#include "sampler_dev.cuh"

using bf16 = __nv_bfloat16;

namespace {

constexpr int FD = 11, FH = 128, FC = 8, FO = 22;
constexpr int N3 = 24;   // layer-3 outputs (22 padded)
// master FP32 layout of one coupling
constexpr int OW1 = 0, OB1 = OW1 + FH * FD, OW2 = OB1 + FH, OB2 = OW2 + FH * FH, OW3 = OB2 + FH,
              OB3 = OW3 + FO * FH, PC = OB3 + FO;
static_assert(PC == LISA_FLOW_PARAMS_PER_COUPLING, "weight layout");
constexpr int NP = FC * PC;
constexpr int TS = 16;     // samples per block
constexpr int NTH = 256;   // eight warps of 16 columns
constexpr int kBatchUnit = 64;  // minibatches are multiples of it
// bfloat16 copies of one coupling in the order of the mma's B fragments (pair_at, single_at):
// the forward layers and the backward ones (transposed)
constexpr int BF1 = 0, BF2 = BF1 + 8 * 256, BF3 = BF2 + 64 * 256, BG3 = BF3 + 12 * 256,
              BG2 = BG3 + 16 * 256, BG1 = BG2 + 64 * 256, BC = BG1 + 8 * 256;
// shared-memory leading dimensions (bf16 elements), padded against bank conflicts
constexpr int LW1 = 24, LH = 136, LGO = 40, LU = 12;
constexpr float kS = 2.0f;  // s = kS tanh(o_s / kS)
constexpr double kLog2Pi = 1.8378770664093454835606594728112353;

__host__ __device__ inline bool keep(int c, int d) {
    switch (c & 3) {
        case 0: return (d & 1) == 0;
        case 1: return (d & 1) == 1;
        case 2: return d < 6;
        default: return d >= 6;
    }
}

// Position of B[k][n] of a K = 16 KS operand: lane (n % 8) 4 + (k % 8) / 2 of the fragment
// (n / 8, k / 16), 16 bytes a lane, which hold two neighbouring n tiles (pair) or k steps (single)
__host__ __device__ inline int pair_at(int k, int n, int KS) {
    const int lane = (n & 7) * 4 + ((k & 7) >> 1);
    return (((n >> 4) * KS + (k >> 4)) * 32 + lane) * 8 + ((n >> 3) & 1) * 4 + ((k >> 3) & 1) * 2 + (k & 1);
}
__host__ __device__ inline int single_at(int k, int n, int KS) {
    const int lane = (n & 7) * 4 + ((k & 7) >> 1);
    return (((n >> 3) * (KS / 2) + (k >> 5)) * 32 + lane) * 8 + ((k >> 4) & 1) * 4 + ((k >> 3) & 1) * 2 + (k & 1);
}

// master weight i of a coupling (not a bias) into both packed copies
__device__ __forceinline__ void pack_weight(bf16 *wb, int i, float v) {
    const bf16 h = __float2bfloat16_rn(v);
    if (i < OB1) {
        const int r = i / FD, k = i % FD;
        wb[BF1 + pair_at(k, r, 1)] = h;
        wb[BG1 + single_at(r, k, 8)] = h;
    } else if (i >= OW2 && i < OB2) {
        const int r = (i - OW2) / FH, k = (i - OW2) % FH;
        wb[BF2 + pair_at(k, r, 8)] = h;
        wb[BG2 + pair_at(r, k, 8)] = h;
    } else if (i >= OW3 && i < OB3) {
        const int r = (i - OW3) / FH, k = (i - OW3) % FH;
        wb[BF3 + single_at(k, r, 8)] = h;
        wb[BG3 + pair_at(r, k, 2)] = h;
    }
}

// ------------------------------------------------------------------ warp GEMMs
__device__ __forceinline__ uint32_t pk(float lo, float hi) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t *>(&v);
}

__device__ __forceinline__ void mma(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
        "{%8,%9}, {%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// A fragment of A[16][16] at p (row-major, leading dimension ld, 16-byte aligned rows)
__device__ __forceinline__ void load_a(uint32_t (&a)[4], const bf16 *p, int ld, int lane) {
    const uint32_t s = (uint32_t)__cvta_generic_to_shared(p + (lane & 15) * ld + (lane >> 4) * 8);
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3])
                 : "r"(s));
}

// S[16][16] at p transposed: as the A fragment of S^T (16 m of 16 k), or as the B fragments
// of two neighbouring n tiles (S = B[k][n])
__device__ __forceinline__ uint4 load_t(const bf16 *p, int ld, int lane, bool as_a) {
    const int q = lane >> 3, r = lane & 7;
    const int kh = as_a ? q >> 1 : q & 1, mh = as_a ? q & 1 : q >> 1;
    const uint32_t s = (uint32_t)__cvta_generic_to_shared(p + (r + 8 * kh) * ld + 8 * mh);
    uint4 v;
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "r"(s));
    return v;
}

__device__ __forceinline__ uint4 frag(const bf16 *wb, int at, int lane) {
    return __ldg(reinterpret_cast<const uint4 *>(wb + at) + lane);
}

// c[2] (16 columns) += A[16][16 KS] B, A in shared memory
template <int KS>
__device__ __forceinline__ void gemm_pair(const bf16 *A, int lda, const uint4 (&b)[KS], float (&c)[2][4],
                                          int lane) {
#pragma unroll
    for (int ks = 0; ks < KS; ks++) {
        uint32_t a[4];
        load_a(a, A + 16 * ks, lda, lane);
        mma(c[0], a, b[ks].x, b[ks].y);
        mma(c[1], a, b[ks].z, b[ks].w);
    }
}

// c (8 columns) += A[16][128] B
__device__ __forceinline__ void gemm_single(const bf16 *A, int lda, const uint4 (&b)[4], float (&c)[4],
                                            int lane) {
#pragma unroll
    for (int k2 = 0; k2 < 4; k2++) {
        uint32_t a[4];
        load_a(a, A + 32 * k2, lda, lane);
        mma(c, a, b[k2].x, b[k2].y);
        load_a(a, A + 32 * k2 + 16, lda, lane);
        mma(c, a, b[k2].z, b[k2].w);
    }
}

// ------------------------------------------------------------------ network
struct FlowView {
    const float *w;
    const bf16 *wb;
    const double *mu, *L;  // mean [11], lower-triangular whitening factor [11][11]
};

// the weights of a coupling that a warp needs in the forward pass
struct Forward {
    uint4 f1[1], f2[8], f3[4];
    float b1[4], b2[4], b3[2];

    __device__ __forceinline__ void load1(const FlowView &f, int c, int warp, int lane) {
        f1[0] = frag(f.wb + (size_t)c * BC, BF1 + warp * 256, lane);
        bias(b1, f.w + (size_t)c * PC + OB1, warp, lane);
    }
    __device__ __forceinline__ void load2(const FlowView &f, int c, int warp, int lane) {
#pragma unroll
        for (int ks = 0; ks < 8; ks++) f2[ks] = frag(f.wb + (size_t)c * BC, BF2 + (warp * 8 + ks) * 256, lane);
        bias(b2, f.w + (size_t)c * PC + OB2, warp, lane);
    }
    __device__ __forceinline__ void load3(const FlowView &f, int c, int warp, int lane) {
        if (warp >= 3) return;
#pragma unroll
        for (int k2 = 0; k2 < 4; k2++) f3[k2] = frag(f.wb + (size_t)c * BC, BF3 + (warp * 4 + k2) * 256, lane);
#pragma unroll
        for (int j = 0; j < 2; j++) {
            const int col = warp * 8 + 2 * (lane & 3) + j;
            b3[j] = col < FO ? __ldg(f.w + (size_t)c * PC + OB3 + col) : 0.0f;
        }
    }
    static __device__ __forceinline__ void bias(float (&b)[4], const float *src, int warp, int lane) {
#pragma unroll
        for (int j = 0; j < 4; j++) b[j] = __ldg(src + warp * 16 + (j >> 1) * 8 + 2 * (lane & 3) + (j & 1));
    }
};

// relu(c + b) of a warp's 16 columns to bf16 rows
__device__ __forceinline__ void put_relu(bf16 *out, const float (&c)[2][4], const float (&b)[4], int warp,
                                         int lane) {
    const int g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int i = 0; i < 2; i++) {
        const int col = warp * 16 + i * 8 + 2 * t;
        *reinterpret_cast<uint32_t *>(out + g * LH + col) =
            pk(fmaxf(c[i][0] + b[2 * i], 0.0f), fmaxf(c[i][1] + b[2 * i + 1], 0.0f));
        *reinterpret_cast<uint32_t *>(out + (g + 8) * LH + col) =
            pk(fmaxf(c[i][2] + b[2 * i], 0.0f), fmaxf(c[i][3] + b[2 * i + 1], 0.0f));
    }
}

// The coupling network on the block's 16 rows: a1 = bf16(relu(W1 a0 + b1)), a2 =
// bf16(relu(W2 a1 + b2)), o = W3 a2 + b3; the weights of coupling cn (if >= 0) are fetched as
// those of this one have been used.  Ends with a block barrier.
__device__ __forceinline__ void net_forward(const FlowView &f, Forward &w, int cn, const bf16 *a0, bf16 *a1,
                                            bf16 *a2, float *o, int warp, int lane) {
    {
        float acc[2][4] = {};
        gemm_pair<1>(a0, LW1, w.f1, acc, lane);
        put_relu(a1, acc, w.b1, warp, lane);
        if (cn >= 0) w.load1(f, cn, warp, lane);
    }
    __syncthreads();
    {
        float acc[2][4] = {};
        gemm_pair<8>(a1, LH, w.f2, acc, lane);
        put_relu(a2, acc, w.b2, warp, lane);
        if (cn >= 0) w.load2(f, cn, warp, lane);
    }
    __syncthreads();
    if (warp < 3) {
        float acc[4] = {};
        gemm_single(a2, LH, w.f3, acc, lane);
        const int g = lane >> 2, col = warp * 8 + 2 * (lane & 3);
        o[g * N3 + col] = acc[0] + w.b3[0];
        o[g * N3 + col + 1] = acc[1] + w.b3[1];
        o[(g + 8) * N3 + col] = acc[2] + w.b3[0];
        o[(g + 8) * N3 + col + 1] = acc[3] + w.b3[1];
        if (cn >= 0) w.load3(f, cn, warp, lane);
    }
    __syncthreads();
}

// thread (row, d): coordinate d of row after coupling c, normalizing (x -> z) or generating
// (z -> x); s is what it was scaled by (kept coordinates: 0)
__device__ __forceinline__ float couple(const float *o, int c, int row, int d, bool gen, float u, float &s) {
    s = 0.0f;
    if (d >= FD || keep(c, d)) return u;
    s = kS * tanhf(o[row * N3 + d] / kS);
    const float tt = o[row * N3 + FD + d];
    return gen ? u * expf(s) + tt : (u - tt) * expf(-s);
}

// thread (row, d): the network's input of coupling c
__device__ __forceinline__ void put_a0(bf16 *a0, int c, int row, int d, float u) {
    a0[row * LW1 + d] = __float2bfloat16_rn(d < FD && keep(c, d) ? u : 0.0f);
}

// a row's sum of s in coupling c, in the order of the coordinates
__device__ __forceinline__ float s_sum(const float *s, int c) {
    float t = 0.0f;
    for (int d = 0; d < FD; d++)
        if (!keep(c, d)) t += s[d];
    return t;
}

// u = L^{-1} (x - mu) by forward substitution (FP64), written as FP32: one thread per row, the
// rows of a block in one warp (an FP64 instruction takes a warp's time, 16 clocks of the SM's
// pipe, however few lanes take part: dealt to 16 threads a row, this took 12 us)
__device__ __forceinline__ void whiten_row(const FlowView &f, const double *x, float *u) {
    double v[FD];
#pragma unroll
    for (int d = 0; d < FD; d++) {
        double acc = x[d] - f.mu[d];
#pragma unroll
        for (int j = 0; j < d; j++) acc -= f.L[d * FD + j] * v[j];
        v[d] = acc / f.L[d * FD + d];
        u[d] = (float)v[d];
    }
}

// sum of the logarithms of the factor's diagonal, in order: a whole warp, result on all lanes
__device__ __forceinline__ double log_det_factor(const double *L, int lane) {
    const double l = log(L[min(lane, FD - 1) * (FD + 1)]);
    double s = 0.0;
    for (int d = 0; d < FD; d++) s += __shfl_sync(0xffffffffu, l, d);
    return s;
}

struct SmemNet {
    alignas(16) bf16 a0[TS * LW1];
    alignas(16) bf16 a1[TS * LH];
    alignas(16) bf16 a2[TS * LH];
    float o[TS * N3];
    float u[TS * LU];
    float s[FC][TS][LU];
    double lsig;
};

// all couplings on the block's rows; u: this thread's coordinate (row threadIdx.x / 16, d =
// threadIdx.x % 16), also left in sm.u.  `w` holds the first coupling's weights, and the
// second pass's first one's (cn2, or -1) on return.
__device__ __forceinline__ float run_couplings(SmemNet &sm, const FlowView &f, Forward &w, float u, bool gen,
                                               int cn2) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, row = threadIdx.x >> 4, d = threadIdx.x & 15;
    put_a0(sm.a0, gen ? FC - 1 : 0, row, d, u);
    __syncthreads();
    for (int k = 0; k < FC; k++) {
        const int c = gen ? FC - 1 - k : k, cn = k + 1 < FC ? (gen ? c - 1 : c + 1) : -1;
        net_forward(f, w, cn >= 0 ? cn : cn2, sm.a0, sm.a1, sm.a2, sm.o, warp, lane);
        float s;
        u = couple(sm.o, c, row, d, gen, u, s);
        if (d < LU) sm.s[c][row][d] = s;
        if (cn >= 0)
            put_a0(sm.a0, cn, row, d, u);
        else if (d < LU)
            sm.u[row * LU + d] = u;
        __syncthreads();
    }
    return u;
}

__device__ __forceinline__ void first_weights(const FlowView &f, Forward &w, int c) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    w.load1(f, c, warp, lane);
    w.load2(f, c, warp, lane);
    w.load3(f, c, warp, lane);
}

// ------------------------------------------------------------------ evaluation
// Both directions for up to 16 rows per block.  Normalizing: in = x, out = z;
// generating: in = z, out = x.  logq = log q(x) in both cases.
__global__ void __launch_bounds__(NTH) flow_eval_kernel(FlowView f, const double *in, int n,
                                                        int gen, double *out, double *logq) {
    __shared__ SmemNet sm;
    Forward w;
    first_weights(f, w, gen ? FC - 1 : 0);
    const int r = threadIdx.x >> 4, d = threadIdx.x & 15, row = blockIdx.x * TS + r;
    const int own = blockIdx.x * TS + threadIdx.x;  // threads 0 .. 15: one row each
    double zz = 0.0;
    if (threadIdx.x < TS) {
        float *u = sm.u + threadIdx.x * LU;
        for (int j = 0; j < LU; j++) u[j] = 0.0f;
        if (own < n) {
            if (gen) {  // all of the input is read here: out may be in
                for (int j = 0; j < FD; j++) {
                    const double zv = in[(size_t)own * FD + j];
                    u[j] = (float)zv;
                    zz += zv * zv;
                }
            } else {
                whiten_row(f, in + (size_t)own * FD, u);
            }
        }
    }
    if (threadIdx.x >= NTH - 32) {
        const double l = log_det_factor(f.L, threadIdx.x & 31);
        if (threadIdx.x == NTH - 1) sm.lsig = l;
    }
    __syncthreads();
    const float u = run_couplings(sm, f, w, d < LU ? sm.u[r * LU + d] : 0.0f, gen != 0, -1);
    if (row < n && d < FD) {
        if (gen) {
            double xv = f.mu[d];  // x = mu + L v
            for (int j = 0; j <= d; j++) xv += f.L[d * FD + j] * (double)sm.u[r * LU + j];
            out[(size_t)row * FD + d] = xv;
        } else if (out) {
            out[(size_t)row * FD + d] = u;
        }
    }
    if (threadIdx.x < TS && own < n) {
        double lq = gen ? -0.5 * zz - 0.5 * FD * kLog2Pi : 0.0;
        for (int k = 0; k < FC; k++) {
            const int c = gen ? FC - 1 - k : k;
            lq -= (double)s_sum(sm.s[c][threadIdx.x], c);
        }
        if (!gen)
            for (int j = 0; j < FD; j++) {
                const double v = sm.u[threadIdx.x * LU + j];
                zz += v * v;
            }
        logq[own] = gen ? lq - sm.lsig : -0.5 * zz - 0.5 * FD * kLog2Pi + lq - sm.lsig;
    }
}

// ------------------------------------------------------------------ training
// Operands of the weight gradients of one coupling and 16 samples (a k step of the
// contraction), as 512-byte fragments: dL/d(pre-activations) of layers 2 and 3 and the inputs
// of layer 1 as A, the inputs of layers 2 and 3 and dL/d(pre-activations) of layer 1 as B.
constexpr int UGZ2 = 0, UGO = 8, UA0 = 10, UA1 = 11, UA2 = 19, UGZ1 = 27, kUnits = 35;
constexpr int kChunkSteps = 128;  // k steps held at a time: 2048 samples, 18 MB
constexpr int kBias = 2 * FH + N3;

struct TrainArgs {
    FlowView f;
    const double *data;     // [n][11]
    long long n;
    int batch;              // rows of this minibatch (multiple of 64)
    int row0;               // first of them in this chunk
    uint32_t k0, k1, round, iter;
    int random_rows;        // 1: Philox minibatch rows; 0: rows 0..batch-1 in order
    uint4 *act;             // [FC][steps][kUnits][32]
    float *bias;            // [steps][FC][kBias]: sums over the step's samples
    double *lossp;          // [steps]
};

struct SmemTrain {
    alignas(16) bf16 a0[FC][TS * LW1];
    alignas(16) bf16 a1[FC][TS * LH];
    alignas(16) bf16 a2[FC][TS * LH];
    alignas(16) bf16 go[TS * LGO];
    alignas(16) bf16 gz2[TS * LH];
    alignas(16) bf16 gz1[TS * LH];
    float o[FC][TS * N3];
    float s[FC][TS][LU];
    float z[TS * LU], gv[TS * LU];  // gv: dL/dv of the current layer's output
    float g3[TS * N3];
    double lrow[TS];
};

// sums over the 16 rows of a warp's 16 columns
__device__ __forceinline__ void column_sums(float *out, float (&v)[2][4], int warp, int lane) {
#pragma unroll
    for (int i = 0; i < 2; i++)
#pragma unroll
        for (int j = 0; j < 2; j++) {
            float s = v[i][j] + v[i][j + 2];
            for (int o = 4; o < 32; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (lane < 4) out[warp * 16 + i * 8 + 2 * lane + j] = s;
        }
}

// masked by the relu's output a (> 0), to bf16 rows
__device__ __forceinline__ void put_masked(bf16 *out, float (&v)[2][4], const bf16 *a, int warp, int lane) {
    const int g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int i = 0; i < 2; i++)
#pragma unroll
        for (int h = 0; h < 2; h++) {
            const int at = (g + 8 * h) * LH + warp * 16 + i * 8 + 2 * t;
            float &v0 = v[i][2 * h], &v1 = v[i][2 * h + 1];
            if (!(__bfloat162float(a[at]) > 0.0f)) v0 = 0.0f;
            if (!(__bfloat162float(a[at + 1]) > 0.0f)) v1 = 0.0f;
            *reinterpret_cast<uint32_t *>(out + at) = pk(v0, v1);
        }
}

// Forward and backward pass of 16 samples: one k step of the weight gradients.
__global__ void __launch_bounds__(NTH) flow_train_kernel(TrainArgs a) {
    extern __shared__ __align__(16) unsigned char smraw[];
    SmemTrain &sm = *reinterpret_cast<SmemTrain *>(smraw);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int row = threadIdx.x >> 4, d = threadIdx.x & 15, step = blockIdx.x, steps = gridDim.x;
    const float inv_n = 1.0f / (float)a.batch;
    const FlowView f = a.f;
    Forward w;
    first_weights(f, w, 0);
    // minibatch rows, whitened
    float u, us[FC];  // coordinate d of every coupling's input
    if (threadIdx.x < TS) {
        const int j = a.row0 + step * TS + threadIdx.x;
        long long idx = j;
        if (a.random_rows) {
            const lisa_smp::U4 q = lisa_smp::philox(a.round, 5u, a.iter, (uint32_t)(j >> 2), a.k0, a.k1);
            idx = (long long)(lisa_smp::unit(q.v[j & 3]) * (double)a.n);
            if (idx > a.n - 1) idx = a.n - 1;
        }
        sm.z[threadIdx.x * LU + FD] = 0.0f;
        whiten_row(f, a.data + idx * FD, sm.z + threadIdx.x * LU);
    }
    __syncthreads();
    u = d < LU ? sm.z[row * LU + d] : 0.0f;
    put_a0(sm.a0[0], 0, row, d, u);
    __syncthreads();
#pragma unroll
    for (int c = 0; c < FC; c++) {
        us[c] = u;
        net_forward(f, w, c + 1 < FC ? c + 1 : -1, sm.a0[c], sm.a1[c], sm.a2[c], sm.o[c], warp, lane);
        float s;
        u = couple(sm.o[c], c, row, d, false, u, s);
        if (d < LU) sm.s[c][row][d] = s;
        if (c + 1 < FC) put_a0(sm.a0[c + 1], c + 1, row, d, u);
        uint4 *act = a.act + ((size_t)c * steps + step) * kUnits * 32 + lane;
        if (warp == 0) act[UA0 * 32] = load_t(sm.a0[c], LW1, lane, true);
        act[(UA1 + warp) * 32] = load_t(sm.a1[c] + 16 * warp, LH, lane, false);
        act[(UA2 + warp) * 32] = load_t(sm.a2[c] + 16 * warp, LH, lane, false);
        __syncthreads();
    }
    // loss and dL/dz = z / batch
    if (d < LU) sm.z[row * LU + d] = u;
    float gv = u * inv_n;  // dL/dv of coordinate d
    uint4 g3[2], g2[8], g1[4];
    auto load3 = [&](int c) {
#pragma unroll
        for (int ks = 0; ks < 2; ks++) g3[ks] = frag(f.wb + (size_t)c * BC, BG3 + (warp * 2 + ks) * 256, lane);
    };
    auto load2 = [&](int c) {
#pragma unroll
        for (int ks = 0; ks < 8; ks++) g2[ks] = frag(f.wb + (size_t)c * BC, BG2 + (warp * 8 + ks) * 256, lane);
    };
    auto load1 = [&](int c) {
        if (warp >= 2) return;
#pragma unroll
        for (int k2 = 0; k2 < 4; k2++) g1[k2] = frag(f.wb + (size_t)c * BC, BG1 + (warp * 4 + k2) * 256, lane);
    };
    load3(FC - 1);
    load2(FC - 1);
    load1(FC - 1);
    __syncthreads();
    if (threadIdx.x < TS) {
        const int r = threadIdx.x;
        float zz = 0.0f, ssum = 0.0f;
        for (int j = 0; j < FD; j++) zz += sm.z[r * LU + j] * sm.z[r * LU + j];
        for (int c = 0; c < FC; c++) ssum += s_sum(sm.s[c][r], c);
        sm.lrow[r] = 0.5 * (double)zz + (double)ssum;
    }
#pragma unroll
    for (int c = FC - 1; c >= 0; c--) {
        float *bias = a.bias + ((size_t)step * FC + c) * kBias;
        // dL/ds, dL/dt of the coupling, and dL/du through the affine map
        {
            float gs = 0.0f, gt = 0.0f;
            if (d < FD && !keep(c, d)) {
                const float th = tanhf(sm.o[c][row * N3 + d] / kS);
                const float s = kS * th;
                const float e = expf(-s);
                const float v = (us[c] - sm.o[c][row * N3 + FD + d]) * e;
                gs = (-gv * v + inv_n) * (1.0f - th * th);
                gt = -gv * e;
                gv = gv * e;
            }
            if (d < FD) {
                sm.go[row * LGO + d] = __float2bfloat16_rn(gs);
                sm.go[row * LGO + FD + d] = __float2bfloat16_rn(gt);
                sm.g3[row * N3 + d] = gs;
                sm.g3[row * N3 + FD + d] = gt;
                sm.gv[row * LU + d] = gv;
            } else {
                *reinterpret_cast<uint32_t *>(sm.go + row * LGO + FO + 2 * (d - FD)) = 0u;
            }
        }
        __syncthreads();
        uint4 *act = a.act + ((size_t)c * steps + step) * kUnits * 32 + lane;
        {  // dL/da2 = go W3, through the relu
            float acc[2][4] = {};
            gemm_pair<2>(sm.go, LGO, g3, acc, lane);
            if (c > 0) load3(c - 1);
            put_masked(sm.gz2, acc, sm.a2[c], warp, lane);
            column_sums(bias + FH, acc, warp, lane);
            if (warp < 2) act[(UGO + warp) * 32] = load_t(sm.go + 16 * warp, LGO, lane, true);
            if (warp == 7 && lane < FO) {
                float t = 0.0f;
                for (int r = 0; r < TS; r++) t += sm.g3[r * N3 + lane];
                bias[2 * FH + lane] = t;
            }
        }
        __syncthreads();
        {  // dL/da1 = gz2 W2, through the relu
            float acc[2][4] = {};
            gemm_pair<8>(sm.gz2, LH, g2, acc, lane);
            if (c > 0) load2(c - 1);
            put_masked(sm.gz1, acc, sm.a1[c], warp, lane);
            column_sums(bias, acc, warp, lane);
            act[(UGZ2 + warp) * 32] = load_t(sm.gz2 + 16 * warp, LH, lane, true);
        }
        __syncthreads();
        act[(UGZ1 + warp) * 32] = load_t(sm.gz1 + 16 * warp, LH, lane, false);
        if (warp < 2) {  // dL/da0 = gz1 W1: reaches the kept coordinates of u
            float acc[4] = {};
            gemm_single(sm.gz1, LH, g1, acc, lane);
            if (c > 0) load1(c - 1);
#pragma unroll
            for (int j = 0; j < 4; j++) {
                const int col = warp * 8 + 2 * (lane & 3) + (j & 1), rr = (lane >> 2) + 8 * (j >> 1);
                if (col < FD && keep(c, col)) sm.gv[rr * LU + col] += acc[j];
            }
        }
        __syncthreads();
        if (d < FD) gv = sm.gv[row * LU + d];
    }
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int r = 0; r < TS; r++) t += sm.lrow[r];
        a.lossp[step] = t / (double)a.batch;
    }
}

struct UpdateArgs {
    const uint4 *act;
    const float *bias;
    const double *lossp;
    int steps;
    float *w, *g, *m, *v;
    bf16 *wb;
    double *loss;
    int first, adam;   // first chunk of the minibatch; Adam step (or the gradient to g)
    float lr, c1, c2;
};

// Adam on the FP32 master weights (Kingma & Ba 2015), then the bf16 copies
__device__ __forceinline__ void update(const UpdateArgs &a, int c, int i, float gi) {
    const size_t at = (size_t)c * PC + i;
    if (!a.first) gi += a.g[at];
    if (!a.adam) {
        a.g[at] = gi;
        return;
    }
    if (!isfinite(gi)) gi = 0.0f;
    const float mi = 0.9f * a.m[at] + 0.1f * gi;
    const float vi = 0.999f * a.v[at] + 0.001f * gi * gi;
    a.m[at] = mi;
    a.v[at] = vi;
    const float wi = a.w[at] - a.lr * (mi / a.c1) / (sqrtf(vi / a.c2) + 1e-8f);
    a.w[at] = wi;
    pack_weight(a.wb + (size_t)c * BC, i, wi);
}

// Weight gradients: jobs 0..7 of a coupling are 16 rows of W2 each, 8 and 9 of W3, 10 is W1
// (transposed), 11 the biases of the hidden layers, 12 those of the outputs and the loss.  The warps take every eighth group of 64 samples
// (four k steps in the accumulator, a minibatch's unit) and add up.
constexpr int kJobs = 13;
__global__ void __launch_bounds__(NTH) flow_update_kernel(UpdateArgs a) {
    extern __shared__ __align__(16) float part[];  // [8][16][128]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, job = blockIdx.x, c = blockIdx.y;
    if (job >= 11) {
        const int i = job == 11 ? threadIdx.x : 2 * FH + threadIdx.x;
        if (i < 2 * FH + FO) {
            float s = 0.0f;
#pragma unroll 16
            for (int k = 0; k < a.steps; k++) s += __ldg(a.bias + ((size_t)k * FC + c) * kBias + i);
            update(a, c, i < FH ? OB1 + i : i < 2 * FH ? OB2 + i - FH : OB3 + i - 2 * FH, s);
        } else if (c == 0 && threadIdx.x == NTH - 1) {
            double t = a.first ? 0.0 : *a.loss;
#pragma unroll 16
            for (int k = 0; k < a.steps; k++) t += __ldg(a.lossp + k);
            *a.loss = t;
        }
        return;
    }
    const int ua = job < 8 ? UGZ2 + job : job < 10 ? UGO + job - 8 : UA0;
    const int ub = job < 8 ? UA1 : job < 10 ? UA2 : UGZ1;
    float sum[16][4] = {};
    for (int k0 = 4 * warp; k0 < a.steps; k0 += 32) {
        float acc[16][4] = {};
#pragma unroll
        for (int k = 0; k < 4; k++) {
            const uint4 *p = a.act + ((size_t)c * a.steps + k0 + k) * kUnits * 32 + lane;
            const uint4 fa = p[ua * 32];
            uint4 fb[8];
#pragma unroll
            for (int i = 0; i < 8; i++) fb[i] = p[(ub + i) * 32];
            const uint32_t av[4] = {fa.x, fa.y, fa.z, fa.w};
#pragma unroll
            for (int i = 0; i < 8; i++) {
                mma(acc[2 * i], av, fb[i].x, fb[i].y);
                mma(acc[2 * i + 1], av, fb[i].z, fb[i].w);
            }
        }
#pragma unroll
        for (int i = 0; i < 16; i++)
#pragma unroll
            for (int j = 0; j < 4; j++) sum[i][j] += acc[i][j];
    }
    const int g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int i = 0; i < 16; i++) {
        float *o = part + warp * 16 * FH + i * 8 + 2 * t;
        *reinterpret_cast<float2 *>(o + g * FH) = make_float2(sum[i][0], sum[i][1]);
        *reinterpret_cast<float2 *>(o + (g + 8) * FH) = make_float2(sum[i][2], sum[i][3]);
    }
    __syncthreads();
    for (int e = threadIdx.x; e < 16 * FH; e += NTH) {
        float s = 0.0f;
#pragma unroll
        for (int k = 0; k < 8; k++) s += part[k * 16 * FH + e];
        const int r = e / FH, n = e % FH;
        if (job < 8)
            update(a, c, OW2 + (16 * job + r) * FH + n, s);
        else if (job < 10) {
            if (16 * (job - 8) + r < FO) update(a, c, OW3 + (16 * (job - 8) + r) * FH + n, s);
        } else if (r < FD)
            update(a, c, OW1 + n * FD + r, s);
    }
}

__global__ void pack_kernel(const float *w, bf16 *wb) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < NP) pack_weight(wb + (size_t)(i / PC) * BC, i % PC, w[i]);
}

// mean of each coordinate (one block per coordinate, FP64)
__global__ void mean_kernel(const double *x, long long n, double *mu) {
    __shared__ double red[256];
    const int d = blockIdx.x;
    double s = 0.0;
    for (long long i = threadIdx.x; i < n; i += blockDim.x) s += x[i * FD + d];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) mu[d] = red[0] / (double)n;
}

// covariance entry (i, j), i >= j, one block each (population normalisation)
__global__ void cov_kernel(const double *x, long long n, const double *mu, double *cov) {
    __shared__ double red[256];
    int b = blockIdx.x, i = 0;
    while (b > i) {
        b -= i + 1;
        i++;
    }
    const int j = b;
    double s = 0.0;
    for (long long r = threadIdx.x; r < n; r += blockDim.x)
        s += (x[r * FD + i] - mu[i]) * (x[r * FD + j] - mu[j]);
    red[threadIdx.x] = s;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        cov[i * FD + j] = red[0] / (double)n;
        cov[j * FD + i] = red[0] / (double)n;
    }
}

// Cholesky factor of the covariance, each pivot floored at 1e-12 of its diagonal entry: one
// warp, lane i holds row i (one thread alone: 41 us, a square root or division after another)
__global__ void cholesky_kernel(const double *cov, double *L) {
    const int i = threadIdx.x;
    double l[FD], row[FD];
#pragma unroll
    for (int j = 0; j < FD; j++) {
        l[j] = 0.0;
        row[j] = i < FD ? cov[i * FD + j] : 0.0;
    }
#pragma unroll
    for (int j = 0; j < FD; j++) {
        double acc = row[j];
#pragma unroll
        for (int k = 0; k < j; k++) acc -= l[k] * __shfl_sync(0xffffffffu, l[k], j);
        const double cjj = __shfl_sync(0xffffffffu, row[j], j);
        const double piv = sqrt(fmax(__shfl_sync(0xffffffffu, acc, j), cjj > 0.0 ? 1e-12 * cjj : 1e-300));
        if (i == j) l[j] = piv;
        if (i > j) l[j] = acc / piv;
    }
    if (i < FD)
#pragma unroll
        for (int j = 0; j < FD; j++) L[i * FD + j] = l[j];
}

// ------------------------------------------------------------------ sampler step
// Independence proposals for the coldest temperature: y = flow(z) with z from Philox
// counters (step, 3, blk, w) by Box-Muller, and log q(x) - log q(y).
__global__ void __launch_bounds__(NTH) flow_propose_kernel(FlowView f, lisa_flowint::FStep a) {
    __shared__ SmemNet sm;
    __shared__ double zlat[TS * FD], qy[TS], px[TS * FD];
    Forward wt;
    first_weights(f, wt, FC - 1);
    const int r = threadIdx.x >> 4, d = threadIdx.x & 15, w = blockIdx.x * TS + r;
    const unsigned step = *a.step;
    // latent draws: threads 0 .. 47, four (three) normals each
    if (threadIdx.x < 3 * TS) {
        const int rr = threadIdx.x % TS, blk = threadIdx.x / TS;
        const lisa_smp::U4 q = lisa_smp::philox(step, 3u, (uint32_t)blk, (uint32_t)(blockIdx.x * TS + rr), a.k0, a.k1);
        for (int p = 0; p < 2; p++) {
            const double u1 = lisa_smp::unit(q.v[2 * p]), u2 = lisa_smp::unit(q.v[2 * p + 1]);
            const double rad = sqrt(-2.0 * log(u1));
            double sn, cs;
            sincos(2.0 * lisa_smp::kPi * u2, &sn, &cs);
            const int at = 4 * blk + 2 * p;
            zlat[rr * FD + at] = rad * cs;
            if (at + 1 < FD) zlat[rr * FD + at + 1] = rad * sn;
        }
    }
    if (threadIdx.x >= NTH - 32) {
        const double l = log_det_factor(f.L, threadIdx.x & 31);
        if (threadIdx.x == NTH - 1) sm.lsig = l;
    }
    __syncthreads();
    float u = run_couplings(sm, f, wt, d < FD ? (float)zlat[r * FD + d] : 0.0f, true, 0);  // generate
    const double lsig = sm.lsig;
    const int own = blockIdx.x * TS + threadIdx.x;  // threads 0 .. 15: one row each
    if (d < FD) {
        double xv = f.mu[d];  // y = mu + L v
        for (int j = 0; j <= d; j++) xv += f.L[d * FD + j] * (double)sm.u[r * LU + j];
        if (w < a.W) a.fy[(size_t)w * FD + d] = xv;
        px[r * FD + d] = xv;
    }
    if (threadIdx.x < TS) {
        double zz = 0.0, lq = 0.0;
        for (int j = 0; j < FD; j++) zz += zlat[threadIdx.x * FD + j] * zlat[threadIdx.x * FD + j];
        for (int c = FC - 1; c >= 0; c--) lq -= (double)s_sum(sm.s[c][threadIdx.x], c);
        qy[threadIdx.x] = -0.5 * zz - 0.5 * FD * kLog2Pi;
        qy[threadIdx.x] += lq - lsig;
    }
    __syncthreads();
    // log q of the current walkers
    if (threadIdx.x < TS) {
        float *v = sm.u + threadIdx.x * LU;
        for (int j = 0; j < LU; j++) v[j] = 0.0f;
        if (own < a.W) whiten_row(f, a.x + (size_t)own * FD, v);
    }
    __syncthreads();
    u = d < LU ? sm.u[r * LU + d] : 0.0f;
    run_couplings(sm, f, wt, u, false, -1);
    if (threadIdx.x < TS && own < a.W) {
        double zz = 0.0, lq = 0.0;
        for (int c = 0; c < FC; c++) lq -= (double)s_sum(sm.s[c][threadIdx.x], c);
        for (int j = 0; j < FD; j++) {
            const double v = sm.u[threadIdx.x * LU + j];
            zz += v * v;
        }
        const double qx = -0.5 * zz - 0.5 * FD * kLog2Pi + lq - lsig;
        a.fq[own] = qx - qy[threadIdx.x];
        double y[FD];
        for (int j = 0; j < FD; j++) y[j] = px[threadIdx.x * FD + j];
        const double py = lisa_smp::ln_prior(y, a.lo, a.hi);
        a.fpy[own] = py;
        if (a.target == LISA_TARGET_GAUSSIAN)
            a.fly[own] = lisa_smp::gauss_lnl(y, a.mean, a.sig);
        else if (isfinite(py))
            lisa_smp::to_physical(y, a.lisa_frame, a.t0, a.fpth + (size_t)own * FD);
        else
            lisa_smp::invalid_params(a.fpth + (size_t)own * FD);
    }
}

// Metropolis-Hastings acceptance of Eq. (13) with the tempered likelihood of the
// coldest temperature and the prior
// log of the MH ratio of flow proposal w with ln L ly (Eq. (13) with the proposal density)
__device__ __forceinline__ double flow_log_ratio(const lisa_flowint::FStep &a, int w, double ly) {
    const double beta = a.betas[0], py = a.fpy[w];
    const double lt = beta > 0.0 ? __dmul_rn(beta, __dsub_rn(ly, a.lnl[w])) : 0.0;
    return __dadd_rn(__dadd_rn(lt, __dsub_rn(py, a.lnp[w])), a.fq[w]);
}

// Screened flow moves: with the first likelihood's ln L, a proposal whose log ratio falls
// below log u by more than beta margin is rejected here (a second likelihood within
// margin of the first would reject it too); every other one, accepted or undecided, is
// sent to the second likelihood, which decides it.  Proposals not sent on get a NaN
// mass, so the second likelihood spends no dense work on them.
__global__ void flow_screen_kernel(lisa_flowint::FStep a) {
    const int w = blockIdx.x * blockDim.x + threadIdx.x;
    if (w >= a.W) return;
    const lisa_smp::U4 q = lisa_smp::philox(*a.step, 4u, 0u, (uint32_t)w, a.k0, a.k1);
    const double py = a.fpy[w];
    const double lr = flow_log_ratio(a, w, a.fly[w]);
    const double lu = log(lisa_smp::unit(q.v[0]));
    const bool send = isfinite(py) && !(lu >= lr + a.betas[0] * a.margin);
    a.fsent[w] = send ? 1 : 0;
    for (int d = 0; d < FD; d++)
        a.fpth2[(size_t)w * FD + d] = (send || d > 0) ? a.fpth[(size_t)w * FD + d] : NAN;
    if (send) atomicAdd(a.facc + 2, 1ULL);
}

__global__ void flow_accept_kernel(lisa_flowint::FStep a) {
    const int w = blockIdx.x * blockDim.x + threadIdx.x;
    if (w >= a.W) return;
    if (*a.err) return;
    if ((a.like_err && *a.like_err) || (a.like_err2 && *a.like_err2)) {
        atomicOr(a.err, 1);
        return;
    }
    if (w == 0) atomicAdd(a.facc + 1, (unsigned long long)a.W);
    const lisa_smp::U4 q = lisa_smp::philox(*a.step, 4u, 0u, (uint32_t)w, a.k0, a.k1);
    if (a.margin > 0.0 && !a.fsent[w]) return;  // rejected by the screen
    const double beta = a.betas[0], py = a.fpy[w];
    const double ly = a.margin > 0.0 ? a.fly2[w] : a.fly[w];
    const double lt = beta > 0.0 ? __dmul_rn(beta, __dsub_rn(ly, a.lnl[w])) : 0.0;
    const double lr = __dadd_rn(__dadd_rn(lt, __dsub_rn(py, a.lnp[w])), a.fq[w]);
    if (isfinite(py) && log(lisa_smp::unit(q.v[0])) < lr) {
        for (int d = 0; d < FD; d++) a.x[(size_t)w * FD + d] = a.fy[(size_t)w * FD + d];
        a.lnl[w] = ly;
        a.lnp[w] = py;
        atomicAdd(a.facc, 1ULL);
    }
}

int train_smem() { return (int)sizeof(SmemTrain); }
int update_smem() { return (int)(sizeof(float) * 8 * 16 * FH); }

}  // namespace

// ------------------------------------------------------------------ host handle
struct lisa_flow {
    int device = 0;
    float *w = nullptr, *g = nullptr, *m = nullptr, *v = nullptr;
    bf16 *wb = nullptr;
    double *mu = nullptr, *L = nullptr, *cov = nullptr, *loss = nullptr;
    uint4 *act = nullptr;      // weight-gradient operands, bias sums and losses of a chunk's k steps
    float *bias = nullptr;
    double *lossp = nullptr;
    int loss_cap = 0, last_iters = 0;
    float *h_grad = nullptr;
    std::string err;
};

namespace {

lisa_status ffail(lisa_flow_t *f, lisa_status st, const std::string &m) {
    if (f) f->err = m;
    else lisa::set_thread_error(m);
    return st;
}

lisa_status fcuda(lisa_flow_t *f, cudaError_t e, const char *what) {
    return ffail(f, e == cudaErrorMemoryAllocation ? LISA_ERR_OOM : LISA_ERR_CUDA,
                 std::string(what) + ": " + cudaGetErrorString(e));
}

#define FCK(call, what)                                   \
    do {                                                  \
        cudaError_t e_ = (call);                          \
        if (e_ != cudaSuccess) return fcuda(f, e_, what); \
    } while (0)

FlowView view(const lisa_flow_t *f) { return {f->w, f->wb, f->mu, f->L}; }

cudaError_t set_smem_limits() {
    cudaError_t e = cudaFuncSetAttribute(flow_train_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, train_smem());
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(flow_update_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, update_smem());
    return e;
}

lisa_status pack(lisa_flow_t *f, cudaStream_t s) {
    pack_kernel<<<(NP + 255) / 256, 256, 0, s>>>(f->w, f->wb);
    FCK(cudaGetLastError(), "pack kernel launch");
    return LISA_OK;
}

lisa_status ensure_loss(lisa_flow_t *f, int iters) {
    if (iters <= f->loss_cap) return LISA_OK;
    if (f->loss) cudaFree(f->loss);
    f->loss = nullptr;
    FCK(cudaMalloc(&f->loss, sizeof(double) * iters), "device allocation (loss history)");
    f->loss_cap = iters;
    return LISA_OK;
}

lisa_status train_iters(lisa_flow_t *f, const double *d_data, int64_t n, int iters, int batch,
                        double lr, uint64_t seed, uint32_t round, cudaStream_t s, int random_rows) {
    lisa_status st = ensure_loss(f, iters);
    if (st != LISA_OK) return st;
    for (int it = 0; it < iters; it++)
        for (int row0 = 0; row0 < batch; row0 += kChunkSteps * TS) {
            const int steps = std::min(kChunkSteps, (batch - row0) / TS), t = it + 1;
            TrainArgs a;
            a.f = view(f);
            a.data = d_data;
            a.n = n;
            a.batch = batch;
            a.row0 = row0;
            a.k0 = (uint32_t)seed;
            a.k1 = (uint32_t)(seed >> 32);
            a.round = round;
            a.iter = (uint32_t)it;
            a.random_rows = random_rows;
            a.act = f->act;
            a.bias = f->bias;
            a.lossp = f->lossp;
            flow_train_kernel<<<steps, NTH, train_smem(), s>>>(a);
            FCK(cudaGetLastError(), "flow training kernel launch");
            UpdateArgs u;
            u.act = f->act;
            u.bias = f->bias;
            u.lossp = f->lossp;
            u.steps = steps;
            u.w = f->w;
            u.g = f->g;
            u.m = f->m;
            u.v = f->v;
            u.wb = f->wb;
            u.loss = f->loss + it;
            u.first = row0 == 0;
            u.adam = lr > 0.0 && row0 + steps * TS == batch;
            u.lr = (float)lr;
            u.c1 = (float)(1.0 - std::pow(0.9, t));
            u.c2 = (float)(1.0 - std::pow(0.999, t));
            flow_update_kernel<<<dim3(kJobs, FC), NTH, update_smem(), s>>>(u);
            FCK(cudaGetLastError(), "flow update kernel launch");
        }
    f->last_iters = iters;
    return LISA_OK;
}

}  // namespace

namespace lisa_flowint {

cudaError_t launch_flow_propose(lisa_flow_t *f, const FStep &a, cudaStream_t s) {
    flow_propose_kernel<<<(a.W + TS - 1) / TS, NTH, 0, s>>>(view(f), a);
    return cudaGetLastError();
}

cudaError_t launch_flow_screen(const FStep &a, cudaStream_t s) {
    flow_screen_kernel<<<(a.W + 127) / 128, 128, 0, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_flow_accept(const FStep &a, cudaStream_t s) {
    flow_accept_kernel<<<(a.W + 127) / 128, 128, 0, s>>>(a);
    return cudaGetLastError();
}

lisa_status flow_train_async(lisa_flow_t *f, const double *d_data, int64_t n, int iters,
                             int batch, double lr, uint64_t seed, uint32_t round, cudaStream_t s) {
    mean_kernel<<<FD, 256, 0, s>>>(d_data, n, f->mu);
    cov_kernel<<<FD * (FD + 1) / 2, 256, 0, s>>>(d_data, n, f->mu, f->cov);
    cholesky_kernel<<<1, 32, 0, s>>>(f->cov, f->L);
    FCK(cudaGetLastError(), "whitening kernel launch");
    FCK(cudaMemsetAsync(f->m, 0, sizeof(float) * NP, s), "cudaMemsetAsync");
    FCK(cudaMemsetAsync(f->v, 0, sizeof(float) * NP, s), "cudaMemsetAsync");
    return train_iters(f, d_data, n, iters, batch, lr, seed, round, s, 1);
}

lisa_status flow_last_loss(lisa_flow_t *f, double *loss, cudaStream_t s) {
    if (f->last_iters < 1) {
        *loss = NAN;
        return LISA_OK;
    }
    FCK(cudaMemcpyAsync(loss, f->loss + f->last_iters - 1, sizeof(double), cudaMemcpyDeviceToHost, s),
        "loss download");
    FCK(cudaStreamSynchronize(s), "cudaStreamSynchronize");
    return LISA_OK;
}

}  // namespace lisa_flowint

extern "C" {

lisa_status lisa_flow_create(uint64_t seed, lisa_flow_t **out) {
    lisa::set_thread_error("");
    if (!out) return ffail(nullptr, LISA_ERR_ARG, "NULL output pointer");
    *out = nullptr;
    lisa_flow_t *f = new lisa_flow();
    lisa_status st = LISA_OK;
    do {
        cudaError_t e = cudaGetDevice(&f->device);
        if (e == cudaSuccess) e = set_smem_limits();
        if (e == cudaSuccess) e = cudaMalloc(&f->w, sizeof(float) * NP);
        if (e == cudaSuccess) e = cudaMalloc(&f->g, sizeof(float) * NP);
        if (e == cudaSuccess) e = cudaMalloc(&f->m, sizeof(float) * NP);
        if (e == cudaSuccess) e = cudaMalloc(&f->v, sizeof(float) * NP);
        if (e == cudaSuccess) e = cudaMalloc(&f->wb, sizeof(bf16) * FC * BC);
        if (e == cudaSuccess) e = cudaMemset(f->wb, 0, sizeof(bf16) * FC * BC);  // the padding
        if (e == cudaSuccess) e = cudaMalloc(&f->act, sizeof(uint4) * 32 * kUnits * FC * kChunkSteps);
        if (e == cudaSuccess) e = cudaMalloc(&f->bias, sizeof(float) * kBias * FC * kChunkSteps);
        if (e == cudaSuccess) e = cudaMalloc(&f->lossp, sizeof(double) * kChunkSteps);
        if (e == cudaSuccess) e = cudaMalloc(&f->mu, sizeof(double) * FD);
        if (e == cudaSuccess) e = cudaMalloc(&f->L, sizeof(double) * FD * FD);
        if (e == cudaSuccess) e = cudaMalloc(&f->cov, sizeof(double) * FD * FD);
        if (e == cudaSuccess) e = cudaMallocHost(&f->h_grad, sizeof(float) * NP);
        if (e != cudaSuccess) {
            st = fcuda(f, e, "flow allocation");
            break;
        }
        // hidden layers uniform in +-sqrt(6 / fan_in) from Philox, zero output layer
        std::vector<float> w(NP, 0.0f);
        const uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
        for (int c = 0; c < FC; c++) {
            float *ws = w.data() + (size_t)c * PC;
            const double lim1 = std::sqrt(6.0 / FD), lim2 = std::sqrt(6.0 / FH);
            for (int i = 0; i < FH * FD; i++) {
                const lisa_smp::U4 q = lisa_smp::philox((uint32_t)c, 1u, (uint32_t)(i >> 2), 0x1Fu, k0, k1);
                ws[OW1 + i] = (float)(lim1 * (2.0 * lisa_smp::unit(q.v[i & 3]) - 1.0));
            }
            for (int i = 0; i < FH * FH; i++) {
                const lisa_smp::U4 q = lisa_smp::philox((uint32_t)c, 2u, (uint32_t)(i >> 2), 0x1Fu, k0, k1);
                ws[OW2 + i] = (float)(lim2 * (2.0 * lisa_smp::unit(q.v[i & 3]) - 1.0));
            }
        }
        st = lisa_flow_set_weights(f, w.data());
        if (st != LISA_OK) break;
        std::vector<double> mu(FD, 0.0), L(FD * FD, 0.0);
        for (int d = 0; d < FD; d++) L[d * FD + d] = 1.0;
        st = lisa_flow_set_whitening(f, mu.data(), L.data());
    } while (0);
    if (st != LISA_OK) {
        lisa::set_thread_error(f->err);
        lisa_flow_destroy(f);
        return st;
    }
    *out = f;
    return LISA_OK;
}

void lisa_flow_destroy(lisa_flow_t *f) {
    if (!f) return;
    cudaSetDevice(f->device);
    cudaDeviceSynchronize();
    for (void *p : {(void *)f->w, (void *)f->g, (void *)f->m, (void *)f->v, (void *)f->wb,
                    (void *)f->mu, (void *)f->L, (void *)f->cov, (void *)f->loss, (void *)f->act,
                    (void *)f->bias, (void *)f->lossp})
        if (p) cudaFree(p);
    if (f->h_grad) cudaFreeHost(f->h_grad);
    delete f;
}

const char *lisa_flow_last_error(const lisa_flow_t *f) { return f ? f->err.c_str() : lisa::thread_error(); }

lisa_status lisa_flow_set_weights(lisa_flow_t *f, const float *w) {
    if (!f) return LISA_ERR_ARG;
    if (!w) return ffail(f, LISA_ERR_ARG, "NULL weights");
    FCK(cudaSetDevice(f->device), "cudaSetDevice");
    FCK(cudaMemcpy(f->w, w, sizeof(float) * NP, cudaMemcpyHostToDevice), "weight upload");
    lisa_status st = pack(f, nullptr);
    if (st != LISA_OK) return st;
    FCK(cudaDeviceSynchronize(), "weight packing");
    return LISA_OK;
}

lisa_status lisa_flow_get_weights(lisa_flow_t *f, float *w) {
    if (!f) return LISA_ERR_ARG;
    if (!w) return ffail(f, LISA_ERR_ARG, "NULL weights");
    FCK(cudaSetDevice(f->device), "cudaSetDevice");
    FCK(cudaDeviceSynchronize(), "cudaDeviceSynchronize");
    FCK(cudaMemcpy(w, f->w, sizeof(float) * NP, cudaMemcpyDeviceToHost), "weight download");
    return LISA_OK;
}

lisa_status lisa_flow_set_whitening(lisa_flow_t *f, const double *mu, const double *L) {
    if (!f) return LISA_ERR_ARG;
    if (!mu || !L) return ffail(f, LISA_ERR_ARG, "NULL whitening");
    double Lc[FD * FD];
    for (int i = 0; i < FD; i++) {
        if (!std::isfinite(mu[i])) return ffail(f, LISA_ERR_ARG, "mu must be finite");
        for (int j = 0; j < FD; j++) {
            const double v = j <= i ? L[i * FD + j] : 0.0;
            if (!std::isfinite(v)) return ffail(f, LISA_ERR_ARG, "L must be finite");
            Lc[i * FD + j] = v;
        }
        if (!(Lc[i * FD + i] > 0.0)) return ffail(f, LISA_ERR_ARG, "L needs a positive diagonal");
    }
    FCK(cudaSetDevice(f->device), "cudaSetDevice");
    FCK(cudaMemcpy(f->mu, mu, sizeof(double) * FD, cudaMemcpyHostToDevice), "upload");
    FCK(cudaMemcpy(f->L, Lc, sizeof(double) * FD * FD, cudaMemcpyHostToDevice), "upload");
    return LISA_OK;
}

lisa_status lisa_flow_get_whitening(lisa_flow_t *f, double *mu, double *L) {
    if (!f) return LISA_ERR_ARG;
    FCK(cudaSetDevice(f->device), "cudaSetDevice");
    FCK(cudaDeviceSynchronize(), "cudaDeviceSynchronize");
    if (mu) FCK(cudaMemcpy(mu, f->mu, sizeof(double) * FD, cudaMemcpyDeviceToHost), "download");
    if (L) FCK(cudaMemcpy(L, f->L, sizeof(double) * FD * FD, cudaMemcpyDeviceToHost), "download");
    return LISA_OK;
}

static lisa_status eval(lisa_flow_t *f, const double *in, int n, int gen, double *out,
                        double *logq, void *stream) {
    if (!f) return LISA_ERR_ARG;
    if (!in || !logq || n < 0 || (gen && !out)) return ffail(f, LISA_ERR_ARG, "NULL pointer or n < 0");
    if (n == 0) return LISA_OK;
    FCK(cudaSetDevice(f->device), "cudaSetDevice");
    flow_eval_kernel<<<(n + TS - 1) / TS, NTH, 0, (cudaStream_t)stream>>>(view(f), in, n, gen, out, logq);
    FCK(cudaGetLastError(), "flow kernel launch");
    return LISA_OK;
}

lisa_status lisa_flow_normalize(lisa_flow_t *f, const double *d_x, int n, double *d_z,
                                double *d_logq, void *stream) {
    return eval(f, d_x, n, 0, d_z, d_logq, stream);
}

lisa_status lisa_flow_generate(lisa_flow_t *f, const double *d_z, int n, double *d_x,
                               double *d_logq, void *stream) {
    return eval(f, d_z, n, 1, d_x, d_logq, stream);
}

lisa_status lisa_flow_gradients(lisa_flow_t *f, const double *d_x, int n, float *grad,
                                double *loss, void *stream) {
    if (!f) return LISA_ERR_ARG;
    if (!d_x || n < kBatchUnit || n % kBatchUnit) return ffail(f, LISA_ERR_ARG, "n must be a positive multiple of 64");
    FCK(cudaSetDevice(f->device), "cudaSetDevice");
    cudaStream_t s = (cudaStream_t)stream;
    lisa_status st = train_iters(f, d_x, n, 1, n, 0.0, 0, 0, s, 0);
    if (st != LISA_OK) return st;
    if (grad) FCK(cudaMemcpyAsync(f->h_grad, f->g, sizeof(float) * NP, cudaMemcpyDeviceToHost, s), "download");
    double l = 0.0;
    FCK(cudaMemcpyAsync(&l, f->loss, sizeof(double), cudaMemcpyDeviceToHost, s), "download");
    FCK(cudaStreamSynchronize(s), "cudaStreamSynchronize");
    if (grad) std::memcpy(grad, f->h_grad, sizeof(float) * NP);
    if (loss) *loss = l;
    return LISA_OK;
}

lisa_status lisa_flow_train(lisa_flow_t *f, const double *d_data, int64_t n, int iters,
                            int batch, double lr, uint64_t seed, uint32_t round, double *loss,
                            void *stream) {
    if (!f) return LISA_ERR_ARG;
    if (!d_data || n < 2 || iters < 1 || batch < kBatchUnit || batch % kBatchUnit || !(lr > 0.0))
        return ffail(f, LISA_ERR_ARG, "need data (n >= 2), iters >= 1, batch a multiple of 64, lr > 0");
    FCK(cudaSetDevice(f->device), "cudaSetDevice");
    cudaStream_t s = (cudaStream_t)stream;
    lisa_status st = lisa_flowint::flow_train_async(f, d_data, n, iters, batch, lr, seed, round, s);
    if (st != LISA_OK) return st;
    if (loss) FCK(cudaMemcpyAsync(loss, f->loss, sizeof(double) * iters, cudaMemcpyDeviceToHost, s), "download");
    FCK(cudaStreamSynchronize(s), "cudaStreamSynchronize");
    return LISA_OK;
}

}  // extern "C"
