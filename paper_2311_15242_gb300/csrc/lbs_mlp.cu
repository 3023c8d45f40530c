// lbs_mlp.cu — the surrogate network: an ensemble of E fully connected
// networks n_in -> width (x depth hidden layers, SiLU) -> n_out (linear),
// trained by mean-squared error with Adam, evaluated with FP32 or bfloat16
// weights.  Every step of training and inference runs in the kernels below.
//
// Definitions (standard, stated here because the paper has no learned part):
//   SiLU(z) = z s(z), s(z) = 1 / (1 + exp(-z)), SiLU'(z) = s(z)(1 + z(1 - s(z)));
//   loss of a member = mean over the minibatch rows and outputs of (y - t)^2;
//   Adam (Kingma & Ba 2015): m <- b1 m + (1-b1) g, v <- b2 v + (1-b2) g^2,
//   theta <- theta - lr (m / (1 - b1^t)) / (sqrt(v / (1 - b2^t)) + eps).
// Parameters of a member: for each layer l = 1..L, W_l (d_l x d_{l-1},
// row-major) then b_l (d_l); members follow each other.
//
// Layout: rows [E][B][d] of inputs and outputs; the minibatch of a member is drawn with
// replacement from the data set by SplitMix64 (Steele, Lea & Flood 2014)
// on (seed, iteration, member, row), so members see different minibatches.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <new>
#include <vector>

#include "../../include/lbs.h"

namespace {

constexpr int kMaxWidth = 128;  // widest layer
constexpr int kMaxLayers = 8;

__host__ __device__ constexpr int up4(int x) { return (x + 3) & ~3; }

struct Shape {
    int L;                        // weight layers
    int d[kMaxLayers + 1];        // d[0] = n_in, ..., d[L] = n_out
    int ld[kMaxLayers + 1];       // widths rounded up to 4 (rows of the scratch arrays)
    long long woff[kMaxLayers + 1], boff[kMaxLayers + 1];  // offsets in a member's vector
    long long P;                  // parameters per member
    // the kernels' own copy of a member's weights, every row and layer on a
    // 16-byte boundary and zero beyond the width: wt the transpose
    // [d_{l-1}][ld_l] that the forward pass multiplies by, wn the weights as
    // they are, [d_l][ld_{l-1}], for the backward pass, bs the biases [ld_l]
    long long wt[kMaxLayers + 1], wn[kMaxLayers + 1], bs[kMaxLayers + 1];
    long long S;                  // floats of that copy per member
    int wmax;                     // floats of its largest layer
};

__device__ __forceinline__ float sigm(float z) { return 1.0f / (1.0f + expf(-z)); }

__device__ __forceinline__ unsigned long long splitmix64(unsigned long long x) {
    x += 0x9E3779B97F4A7C15ull;
    x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
    x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
    return x ^ (x >> 31);
}

// the copy of the parameters that the kernels multiply by (Shape::wt, wn,
// bs); BF16: the values rounded to bfloat16 (exact as floats)
template <bool BF16>
__global__ void k_copy_weights(const float *p, Shape s, int E, float *W) {
    const long long n = (long long)E * s.P;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n;
         k += (long long)gridDim.x * blockDim.x) {
        const long long e = k / s.P, q = k - e * s.P;
        int l = 1;
        while (l < s.L && q >= s.woff[l + 1]) l++;
        float v = p[k];
        if (BF16) v = __bfloat162float(__float2bfloat16_rn(v));
        float *w = W + e * s.S;
        if (q >= s.boff[l]) {
            w[s.bs[l] + (q - s.boff[l])] = v;
        } else {
            const int r = (int)(q - s.woff[l]), o = r / s.d[l - 1], i = r - o * s.d[l - 1];
            w[s.wt[l] + (long long)i * s.ld[l] + o] = v;
            if (!BF16) w[s.wn[l] + (long long)o * s.ld[l - 1] + i] = v;
        }
    }
}

// ---------------------------------------------------------------------------
// Layer products.  A block holds ROWS rows of one member in shared memory as
// act[k][row] (row stride RS) and one layer's weights as w[k][ldw]; a thread
// keeps a 4 C x 4 tile of the product in registers (C chunks of 4 rows, 4
// outputs), so that a step of k costs C + 1 16-byte shared loads, four
// wavefronts a warp each, for 16 C multiply-adds: at C = 2 the loads take 12
// cycles of the SM's shared memory and the multiply-adds 8 of its FP32 pipes.
// (8 x 8 tiles would balance them, but leave 8 warps an SM, too few to hide the
// loads: 40,000 rows 0.44 -> 0.54 ms.)  ROWS = 64 (C = 2) serves inference, where
// there are enough rows to fill the chip; ROWS = 16 (C = 1) serves training and
// short batches, where the minibatch of every member must spread over many
// blocks; its threads split k in two halves, since 128 threads alone leave the
// schedulers idle.
// ---------------------------------------------------------------------------
template <int ROWS>
struct Tile {
    static constexpr int NT = 256;                   // threads
    static constexpr int C = ROWS == 64 ? 2 : 1;     // row chunks of a thread
    static constexpr int KS = ROWS == 64 ? 1 : 2;    // ways k is split
    static constexpr int RG = ROWS / (4 * C);        // row groups
    static constexpr int RS = ROWS + 4;              // row stride of act
    static_assert(NT / KS == RG * (kMaxWidth / 4), "a thread has one tile of the widest layer");
};

__device__ __forceinline__ void cp16(float *dst, const float *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                     (unsigned)__cvta_generic_to_shared(dst)),
                 "l"(src)
                 : "memory");
}
// start the copy of n floats (a multiple of 4) as one group
__device__ __forceinline__ void start_copy(float *dst, const float *src, int n) {
    for (int q = threadIdx.x * 4; q < n; q += blockDim.x * 4) cp16(dst + q, src + q);
    asm volatile("cp.async.commit_group;" ::: "memory");
}
template <int N>
__device__ __forceinline__ void wait_copies() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

template <int ROWS>
__device__ __forceinline__ void product(const float *act, const float *w, int ldw, int k0, int k1,
                                        int tr, int to, float (&acc)[4 * Tile<ROWS>::C][4]) {
    using T = Tile<ROWS>;
#pragma unroll
    for (int r = 0; r < 4 * T::C; r++)
#pragma unroll
        for (int j = 0; j < 4; j++) acc[r][j] = 0.0f;
#pragma unroll 4
    for (int k = k0; k < k1; k++) {
        const float4 wv = *(const float4 *)(w + k * ldw + 4 * to);
#pragma unroll
        for (int c = 0; c < T::C; c++) {
            const float4 a = *(const float4 *)(act + k * T::RS + c * 4 * T::RG + 4 * tr);
            const float av[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
            for (int r = 0; r < 4; r++) {
                acc[4 * c + r][0] = fmaf(av[r], wv.x, acc[4 * c + r][0]);
                acc[4 * c + r][1] = fmaf(av[r], wv.y, acc[4 * c + r][1]);
                acc[4 * c + r][2] = fmaf(av[r], wv.z, acc[4 * c + r][2]);
                acc[4 * c + r][3] = fmaf(av[r], wv.w, acc[4 * c + r][3]);
            }
        }
    }
}

// an output layer of at most kNarrow outputs: thread (row, part of k), the
// parts added through `part` (NT kNarrow floats); out[row * ldo + o] + bias.
// (With the tiles of `product` a handful of threads would walk all of k.)
constexpr int kNarrow = 8;
template <int ROWS>
__device__ __forceinline__ void product_narrow(const float *act, const float *w, int ldw, int kn,
                                               float *part, float (&sum)[kNarrow]) {
    using T = Tile<ROWS>;
    constexpr int NP = T::NT / ROWS;
    const int row = threadIdx.x % ROWS, ks = threadIdx.x / ROWS;
    const int per = (kn + NP - 1) / NP, k0 = ks * per, k1 = min(kn, k0 + per);
#pragma unroll
    for (int j = 0; j < kNarrow; j++) sum[j] = 0.0f;
    for (int k = k0; k < k1; k++) {
        const float a = act[k * T::RS + row];
#pragma unroll
        for (int j = 0; j < kNarrow; j++)
            if (j < ldw) sum[j] = fmaf(a, w[k * ldw + j], sum[j]);
    }
#pragma unroll
    for (int j = 0; j < kNarrow; j++) part[j * T::NT + threadIdx.x] = sum[j];
    __syncthreads();
    // (the first ROWS threads hold the sums)
    if (ks == 0) {
#pragma unroll
        for (int j = 0; j < kNarrow; j++) {
            sum[j] = part[j * T::NT + row];
            for (int q = 1; q < NP; q++) sum[j] += part[j * T::NT + q * ROWS + row];
        }
    }
}

// outputs of the whole network for ROWS rows of one member (grid: row tiles,
// members): every layer in shared memory, one layer's weights at a time.
// x [B][d_0] of the member (xstride apart; 0: the same rows for every
// member), y [E][B][d_L].  Bound by the FP32 multiply-adds (2 W flops a row
// and member).  With a launch a layer, activations through global memory and
// uncoalesced weights, 40,000 rows of the 5-128-128-128-2 ensemble of 5 took
// 6.38 ms (predict, 40 chunks of 4 launches); now 0.44 ms, 0.37 of it here.
template <int ROWS>
__global__ void __launch_bounds__(Tile<ROWS>::NT, 2)
    k_net_forward(const float *__restrict__ W, Shape s, const float *__restrict__ x,
                  long long xstride, int B, float *__restrict__ y) {
    using T = Tile<ROWS>;
    extern __shared__ __align__(16) float sm[];
    float *w = sm, *act = w + s.wmax, *part = act + kMaxWidth * T::RS;
    const int e = blockIdx.y, r0 = blockIdx.x * ROWS, t = threadIdx.x;
    const int g = T::KS == 1 ? 0 : t / (T::NT / T::KS), tt = t - g * (T::NT / T::KS);
    const int tr = tt % T::RG, to = tt / T::RG;
    W += e * s.S;
    x += e * xstride;
    start_copy(w, W + s.wt[1], s.d[0] * s.ld[1]);
    for (int q = t; q < ROWS * s.d[0]; q += T::NT) {
        const int r = q / s.d[0], i = q - r * s.d[0];
        act[i * T::RS + r] = r0 + r < B ? x[(long long)(r0 + r) * s.d[0] + i] : 0.0f;
    }
    for (int l = 1; l <= s.L; l++) {
        wait_copies<0>();
        __syncthreads();
        const int kn = s.d[l - 1], ldw = s.ld[l];
        const float *bias = W + s.bs[l];
        if (l == s.L && ldw <= kNarrow) {
            float sum[kNarrow];
            product_narrow<ROWS>(act, w, ldw, kn, part, sum);
            if (t < ROWS && r0 + t < B)
#pragma unroll
                for (int j = 0; j < kNarrow; j++)
                    if (j < s.d[l]) y[((long long)e * B + r0 + t) * s.d[l] + j] = sum[j] + bias[j];
            return;
        }
        float acc[4 * T::C][4];
        const bool on = 4 * to < ldw;
        const int kh = T::KS == 1 ? kn : (kn + 1) / 2;
        if (on) product<ROWS>(act, w, ldw, g ? kh : 0, g ? kn : kh, tr, to, acc);
        if (T::KS == 2) {
            if (on && g == 1)
#pragma unroll
                for (int r = 0; r < 4; r++)
                    *(float4 *)(part + (r * (T::NT / 2) + tt) * 4) =
                        make_float4(acc[r][0], acc[r][1], acc[r][2], acc[r][3]);
            __syncthreads();
            if (on && g == 0)
#pragma unroll
                for (int r = 0; r < 4; r++) {
                    const float4 o = *(const float4 *)(part + (r * (T::NT / 2) + tt) * 4);
                    acc[r][0] += o.x;
                    acc[r][1] += o.y;
                    acc[r][2] += o.z;
                    acc[r][3] += o.w;
                }
        } else {
            __syncthreads();
        }
        // (every thread is past its reads of act and w)
        if (l < s.L) start_copy(w, W + s.wt[l + 1], s.d[l] * s.ld[l + 1]);
        if (!on || g) continue;
        const float4 bv = *(const float4 *)(bias + 4 * to);
        const float bj[4] = {bv.x, bv.y, bv.z, bv.w};
#pragma unroll
        for (int c = 0; c < T::C; c++)
#pragma unroll
            for (int j = 0; j < 4; j++) {
                float v[4];
#pragma unroll
                for (int r = 0; r < 4; r++) {
                    const float z = acc[4 * c + r][j] + bj[j];
                    v[r] = l < s.L ? z * sigm(z) : z;
                }
                if (l < s.L) {
                    *(float4 *)(act + (4 * to + j) * T::RS + c * 4 * T::RG + 4 * tr) =
                        make_float4(v[0], v[1], v[2], v[3]);
                } else if (4 * to + j < s.d[l]) {
#pragma unroll
                    for (int r = 0; r < 4; r++) {
                        const int row = r0 + c * 4 * T::RG + 4 * tr + r;
                        if (row < B) y[((long long)e * B + row) * s.d[l] + 4 * to + j] = v[r];
                    }
                }
            }
    }
}

// ---------------------------------------------------------------------------
// Training: two launches an iteration.  k_net_pass draws (or reads) 16 rows
// of a member's minibatch, runs them forward and back through all layers in
// shared memory (the next layer's weights arrive by asynchronous copies while
// the present one is multiplied) and leaves the activations A_l and dL/dZ_l;
// k_net_update forms a 32 x 32 tile of a layer's gradient over the whole
// minibatch and, in training, takes Adam's step for it and renews the kernels'
// copy of those weights.  For 5 members of 5-128-128-128-2 at 256 rows the 14
// launches of one kernel a layer and direction, whose weight gradients walked
// the minibatch row by row, took 356 us an iteration; the two take 42.
// ---------------------------------------------------------------------------
struct Bufs {
    float *A[kMaxLayers + 1];   // activations [E][B][ld_l], l = 0 .. L - 1
    float *dZ[kMaxLayers + 1];  // dL/dZ_l [E][B][ld_l], l = 1 .. L
};

constexpr int kTrainRows = 16;

// floats of shared memory of k_net_pass
__host__ __device__ __forceinline__ size_t pass_floats(const Shape &s) {
    using T = Tile<kTrainRows>;
    size_t hid = 0;
    for (int l = 1; l < s.L; l++) hid += (size_t)s.ld[l] * T::RS;
    return 2 * (size_t)s.wmax + kMaxWidth * T::RS + kNarrow * T::NT + hid +
           (size_t)kTrainRows * s.ld[s.L];
}

// X, Y: the data set, whose row r of `ndata` is drawn for (seed, iter, member,
// row) when ndata > 0; else the member's own rows [E][B][.].  lossp: the
// block's part of the sum of squared errors, [E][gridDim.x].
__global__ void __launch_bounds__(Tile<kTrainRows>::NT)
    k_net_pass(const float *__restrict__ W, Shape s, const float *__restrict__ X,
               const float *__restrict__ Y, int ndata, int B, unsigned long long seed,
               long long iter, Bufs b, double *lossp) {
    using T = Tile<kTrainRows>;
    constexpr int RS = T::RS, HT = T::NT / 2;
    extern __shared__ __align__(16) float sm[];
    float *wbuf[2] = {sm, sm + s.wmax};
    float *act = sm + 2 * s.wmax, *part = act + kMaxWidth * RS, *der = part + kNarrow * T::NT;
    float *tgt = der;  // (set below: after the derivatives of every hidden layer)
    for (int l = 1; l < s.L; l++) tgt += s.ld[l] * RS;
    __shared__ int src[kTrainRows];
    __shared__ double sq[T::NT / 32];
    const int e = blockIdx.y, r0 = blockIdx.x * kTrainRows, t = threadIdx.x;
    const int E = gridDim.y;
    const int g = t / HT, tt = t - g * HT, tr = tt % T::RG, to = tt / T::RG;
    W += e * s.S;
    start_copy(wbuf[0], W + s.wt[1], s.d[0] * s.ld[1]);
    start_copy(wbuf[1], W + s.wt[2], s.d[1] * s.ld[2]);  // (there are two layers at least)
    if (t < kTrainRows) {
        long long r = -1;
        if (r0 + t < B) {
            if (ndata > 0) {
                const unsigned long long key =
                    ((unsigned long long)iter * E + e) * (unsigned long long)B + (r0 + t);
                r = (long long)(splitmix64(seed ^ splitmix64(key)) % (unsigned long long)ndata);
            } else {
                r = t;
            }
        }
        src[t] = (int)r;
    }
    __syncthreads();
    const long long base = ndata > 0 ? 0 : (long long)e * B + r0;
    const int d0 = s.d[0], dL = s.d[s.L], ldL = s.ld[s.L];
    for (int q = t; q < kTrainRows * s.ld[0]; q += T::NT) {
        const int r = q / s.ld[0], i = q - r * s.ld[0];
        const float v = src[r] >= 0 && i < d0 ? X[(base + src[r]) * d0 + i] : 0.0f;
        if (i < d0) act[i * RS + r] = v;
        if (r0 + r < B) b.A[0][((long long)e * B + r0 + r) * s.ld[0] + i] = v;
    }
    for (int q = t; q < kTrainRows * ldL; q += T::NT) {
        const int r = q / ldL, o = q - r * ldL;
        tgt[q] = src[r] >= 0 && o < dL ? Y[(base + src[r]) * dL + o] : 0.0f;
    }
    const float sc = 2.0f / float((long long)B * dL);
    // passes 0 .. L - 1 forward (layers 1 .. L), L .. 2 L - 2 back (layers L .. 2)
    float *dl = der;  // derivatives of the present hidden layer
    for (int p = 0; p < 2 * s.L - 1; p++) {
        const bool fwd = p < s.L;
        const int l = fwd ? p + 1 : 2 * s.L - p;
        const int kn = fwd ? s.d[l - 1] : s.d[l], ldw = fwd ? s.ld[l] : s.ld[l - 1];
        const float *w = wbuf[p & 1];
        wait_copies<1>();
        __syncthreads();
        double err = 0.0;
        const bool narrow = fwd && l == s.L && ldw <= kNarrow;
        float acc[4][4];
        float sum[kNarrow];
        const bool on = 4 * to < ldw;
        if (narrow) {
            product_narrow<kTrainRows>(act, w, ldw, kn, part, sum);
        } else {
            const int kh = (kn + 1) / 2;
            if (on) {
                product<kTrainRows>(act, w, ldw, g ? kh : 0, g ? kn : kh, tr, to, acc);
                // group 0 finishes rows 0, 1 of the tile, group 1 rows 2, 3
#pragma unroll
                for (int r = 0; r < 2; r++) {
                    const int o = g ? r : r + 2;
                    *(float4 *)(part + ((2 * g + r) * HT + tt) * 4) =
                        make_float4(acc[o][0], acc[o][1], acc[o][2], acc[o][3]);
                }
            }
        }
        __syncthreads();
        // the weights of pass p + 2 into the buffer of this pass
        {
            const int n = p + 2;
            if (n < s.L)
                start_copy(wbuf[p & 1], W + s.wt[n + 1], s.d[n] * s.ld[n + 1]);
            else if (n < 2 * s.L - 1)
                start_copy(wbuf[p & 1], W + s.wn[2 * s.L - n],
                           s.d[2 * s.L - n] * s.ld[2 * s.L - n - 1]);
            else
                start_copy(wbuf[p & 1], W, 0);
        }
        if (narrow) {
            if (t < kTrainRows) {
                const bool in = r0 + t < B;
                float dz[kNarrow];
#pragma unroll
                for (int j = 0; j < kNarrow; j++) {
                    dz[j] = 0.0f;
                    if (j < dL && in) {
                        const float d = (sum[j] + W[s.bs[l] + j]) - tgt[t * ldL + j];
                        err += double(d) * double(d);
                        dz[j] = sc * d;
                    }
                    if (j < ldL) {
                        act[j * RS + t] = dz[j];
                        if (in) b.dZ[l][((long long)e * B + r0 + t) * ldL + j] = dz[j];
                    }
                }
            }
        } else if (on) {
            float v[2][4];
#pragma unroll
            for (int r = 0; r < 2; r++) {
                const float4 o = *(const float4 *)(part + ((2 * (1 - g) + r) * HT + tt) * 4);
                const int k = g ? r + 2 : r;
                v[r][0] = acc[k][0] + o.x;
                v[r][1] = acc[k][1] + o.y;
                v[r][2] = acc[k][2] + o.z;
                v[r][3] = acc[k][3] + o.w;
            }
            const int row = 4 * tr + 2 * g;  // of the tile's rows 2 g, 2 g + 1
            float *dst = nullptr;            // of A_l or dZ_{l-1}, its row stride
            if (fwd) {
                const float4 bv = *(const float4 *)(W + s.bs[l] + 4 * to);
                const float bj[4] = {bv.x, bv.y, bv.z, bv.w};
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    float dv[2];
#pragma unroll
                    for (int r = 0; r < 2; r++) {
                        const float z = v[r][j] + bj[j];
                        if (l < s.L) {
                            const float sg = sigm(z);
                            v[r][j] = z * sg;
                            dv[r] = sg * (1.0f + z * (1.0f - sg));
                        } else {
                            float d = 0.0f;
                            if (4 * to + j < dL && r0 + row + r < B)
                                d = z - tgt[(row + r) * ldL + 4 * to + j];
                            err += double(d) * double(d);
                            v[r][j] = sc * d;
                        }
                    }
                    if (l < s.L)
                        *(float2 *)(dl + (4 * to + j) * RS + row) = make_float2(dv[0], dv[1]);
                }
                dst = l < s.L ? b.A[l] : b.dZ[l];
            } else {
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    const float2 dv = *(const float2 *)(dl + (4 * to + j) * RS + row);
                    v[0][j] *= dv.x;
                    v[1][j] *= dv.y;
                }
                dst = b.dZ[l - 1];
            }
#pragma unroll
            for (int j = 0; j < 4; j++)
                *(float2 *)(act + (4 * to + j) * RS + row) = make_float2(v[0][j], v[1][j]);
#pragma unroll
            for (int r = 0; r < 2; r++)
                if (r0 + row + r < B)
                    *(float4 *)(dst + ((long long)e * B + r0 + row + r) * ldw + 4 * to) =
                        make_float4(v[r][0], v[r][1], v[r][2], v[r][3]);
        }
        if (fwd && l < s.L - 1) dl += s.ld[l] * RS;
        if (!fwd && l > 2) dl -= s.ld[l - 2] * RS;
        if (fwd && l == s.L) {
            // the block's squared errors, in a fixed order
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) err += __shfl_down_sync(0xffffffffu, err, o);
            if ((t & 31) == 0) sq[t >> 5] = err;
            __syncthreads();
            if (t == 0) {
                double q = 0.0;
                for (int k = 0; k < T::NT / 32; k++) q += sq[k];
                lossp[(long long)e * gridDim.x + blockIdx.x] = q;
            }
        }
    }
    wait_copies<0>();
}

// loss of every member from its blocks' sums, in order
__global__ void k_loss_sum(const double *lossp, int tiles, long long n, double *loss) {
    const int e = blockIdx.x;
    double s = 0.0;
    for (int k = threadIdx.x; k < tiles; k += 32) s += lossp[(long long)e * tiles + k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (threadIdx.x == 0) loss[e] = s / double(n);
}

struct Adam {
    int on;
    float lr, b1, b2, eps, c1, c2;
};

__device__ __forceinline__ float adam_one(const Adam &a, float p, float g, float &m, float &v) {
    m = a.b1 * m + (1.0f - a.b1) * g;
    v = a.b2 * v + (1.0f - a.b2) * g * g;
    return p - a.lr * (m / a.c1) / (sqrtf(v / a.c2) + a.eps);
}

constexpr int kUpTile = 32, kUpRows = 128;  // gradient tile, rows staged at a time

// grid: (32 x 32 tiles of every layer's dW, members), 256 threads.  The
// threads are four groups of 64; a group takes every fourth row of the
// minibatch with a 4 x 4 tile a thread (two 16-byte shared loads for 16
// multiply-adds), and the groups' sums are added through shared memory.  The
// block of a row of tiles' first column also sums the biases' gradient.
__global__ void __launch_bounds__(256)
    k_net_update(Shape s, int B, Bufs b, Adam ad, float *params, float *grad, float *mom, float *var,
                 float *W) {
    __shared__ __align__(16) float zs[kUpRows][kUpTile], as[kUpRows][kUpTile];
    __shared__ float tp[kUpTile][kUpTile + 1];
    __shared__ float bsum[8][kUpTile];
    const int e = blockIdx.y, t = threadIdx.x;
    int l = 1, k = blockIdx.x, nti = 1;
    for (;; l++) {
        nti = (s.d[l - 1] + kUpTile - 1) / kUpTile;
        const int n = nti * ((s.d[l] + kUpTile - 1) / kUpTile);
        if (k < n) break;
        k -= n;
    }
    const int o0 = (k / nti) * kUpTile, i0 = (k % nti) * kUpTile;
    const int ldz = s.ld[l], lda = s.ld[l - 1];
    const float *dz = b.dZ[l] + (long long)e * B * ldz, *a = b.A[l - 1] + (long long)e * B * lda;
    const int g = t >> 6, q = t & 63, og = q & 7, ig = q >> 3;
    float acc[4][4];
#pragma unroll
    for (int r = 0; r < 4; r++)
#pragma unroll
        for (int j = 0; j < 4; j++) acc[r][j] = 0.0f;
    float bacc = 0.0f;  // (thread t: output t % 32, rows t / 32 mod 8)
    for (int b0 = 0; b0 < B; b0 += kUpRows) {
        __syncthreads();
        // 8 threads a row, 32 rows a turn
        float4 zv[kUpRows / 32], av[kUpRows / 32];
#pragma unroll
        for (int u = 0; u < kUpRows / 32; u++) {
            const int r = b0 + u * 32 + (t >> 3), c = (t & 7) * 4;
            zv[u] = av[u] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            if (r < B && o0 + c < ldz) zv[u] = *(const float4 *)(dz + (long long)r * ldz + o0 + c);
            if (r < B && i0 + c < lda) av[u] = *(const float4 *)(a + (long long)r * lda + i0 + c);
        }
#pragma unroll
        for (int u = 0; u < kUpRows / 32; u++) {
            *(float4 *)&zs[u * 32 + (t >> 3)][(t & 7) * 4] = zv[u];
            *(float4 *)&as[u * 32 + (t >> 3)][(t & 7) * 4] = av[u];
        }
        __syncthreads();
#pragma unroll 8
        for (int r = g; r < kUpRows; r += 4) {
            const float4 z4 = *(const float4 *)&zs[r][4 * og], a4 = *(const float4 *)&as[r][4 * ig];
            const float z[4] = {z4.x, z4.y, z4.z, z4.w}, v[4] = {a4.x, a4.y, a4.z, a4.w};
#pragma unroll
            for (int x = 0; x < 4; x++)
#pragma unroll
                for (int j = 0; j < 4; j++) acc[x][j] = fmaf(z[x], v[j], acc[x][j]);
        }
        if (i0 == 0)
            for (int r = t >> 5; r < kUpRows; r += 8) bacc += zs[r][t & 31];
    }
    __syncthreads();
    // the four groups' sums, in order: group g leaves its tile in the staging
    // rows, thread t then adds elements t, t + 256, ... of the 32 x 32 tile
    float *red = &zs[0][0];  // [4][32][32]
#pragma unroll
    for (int x = 0; x < 4; x++)
        *(float4 *)(red + (g * kUpTile + 4 * og + x) * kUpTile + 4 * ig) =
            make_float4(acc[x][0], acc[x][1], acc[x][2], acc[x][3]);
    if (i0 == 0) bsum[t >> 5][t & 31] = bacc;
    __syncthreads();
    const long long pb = (long long)e * s.P;
    float *We = W + e * s.S;
#pragma unroll
    for (int u = 0; u < 4; u++) {
        const int idx = t + 256 * u, ol = idx >> 5, il = idx & 31, o = o0 + ol, i = i0 + il;
        if (o < s.d[l] && i < s.d[l - 1]) {
            const float gr = (red[idx] + red[idx + 1024]) + (red[idx + 2048] + red[idx + 3072]);
            const long long c = pb + s.woff[l] + (long long)o * s.d[l - 1] + i;
            grad[c] = gr;
            if (ad.on) {
                float m = mom[c], v = var[c];
                const float p = adam_one(ad, params[c], gr, m, v);
                mom[c] = m;
                var[c] = v;
                params[c] = p;
                We[s.wn[l] + (long long)o * lda + i] = p;
                tp[il][ol] = p;
            }
        }
    }
    if (i0 == 0 && t < kUpTile && o0 + t < s.d[l]) {
        float gr = 0.0f;
#pragma unroll
        for (int u = 0; u < 8; u++) gr += bsum[u][t];
        const long long c = pb + s.boff[l] + o0 + t;
        grad[c] = gr;
        if (ad.on) {
            float m = mom[c], v = var[c];
            const float p = adam_one(ad, params[c], gr, m, v);
            mom[c] = m;
            var[c] = v;
            params[c] = p;
            We[s.bs[l] + o0 + t] = p;
        }
    }
    if (!ad.on) return;
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 4; u++) {
        const int idx = t + 256 * u, il = idx >> 5, ol = idx & 31;
        if (o0 + ol < s.d[l] && i0 + il < s.d[l - 1])
            We[s.wt[l] + (long long)(i0 + il) * ldz + o0 + ol] = tp[il][ol];
    }
}

__global__ void k_adam(float *p, const float *g, float *m, float *v, long long n, Adam a) {
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n;
         k += (long long)gridDim.x * blockDim.x) {
        float mk = m[k], vk = v[k];
        p[k] = adam_one(a, p[k], g[k], mk, vk);
        m[k] = mk;
        v[k] = vk;
    }
}

// ensemble mean and standard deviation (population) over the E members
__global__ void k_stats(const float *Y, int E, long long n, float *mean, float *sd) {
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n;
         k += (long long)gridDim.x * blockDim.x) {
        double s = 0, s2 = 0;
        for (int e = 0; e < E; e++) s += Y[(long long)e * n + k];
        const double mu = s / E;
        for (int e = 0; e < E; e++) {
            const double d = Y[(long long)e * n + k] - mu;
            s2 += d * d;
        }
        mean[k] = float(mu);
        sd[k] = float(sqrt(s2 / E));
    }
}

// Glorot-uniform weights, zero biases, from SplitMix64 on (seed, index)
__global__ void k_init(float *p, long long n, const long long *woff, const long long *boff,
                       const int *d, int L, long long P, unsigned long long seed) {
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n;
         k += (long long)gridDim.x * blockDim.x) {
        const long long q = k % P;
        float val = 0.0f;
        for (int l = 1; l <= L; l++) {
            if (q >= woff[l] && q < boff[l]) {
                const float a = sqrtf(6.0f / float(d[l - 1] + d[l]));
                const unsigned long long r = splitmix64(seed ^ splitmix64((unsigned long long)k));
                const float u = float((r >> 40) * (1.0 / 16777216.0));  // [0, 1), 24 bits
                val = (2.0f * u - 1.0f) * a;
            }
        }
        p[k] = val;
    }
}

}  // namespace

struct lbs_mlp {
    int E = 0, B = 0;
    Shape s;
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    float *params = nullptr, *grad = nullptr, *m = nullptr, *v = nullptr;
    // the kernels' copies of the weights (Shape::wt ...): as they are, and
    // rounded to bfloat16; valid until the parameters change
    float *W = nullptr, *Wbf = nullptr;
    bool w_valid = false, bf_valid = false;
    Bufs bufs = {};
    float *x = nullptr, *y = nullptr, *T = nullptr, *stats = nullptr;
    double *lossp = nullptr, *loss = nullptr;
    // workspace of predict for more rows than max_batch (rows it holds)
    float *px = nullptr, *py = nullptr, *pstats = nullptr;
    int prows = 0;
    float *X = nullptr, *Yd = nullptr;
    int ndata = 0;
    int sms = 1;
    long long t = 0;  // Adam steps taken
    char err[512] = {0};

    void drop_predict() {
        cudaFree(px);
        cudaFree(py);
        cudaFree(pstats);
        px = py = pstats = nullptr;
        prows = 0;
    }
    ~lbs_mlp() {
        if (stream) cudaStreamSynchronize(stream);
        float *fl[] = {params, grad, m, v, W, Wbf, x, y, T, stats, X, Yd};
        for (float *p : fl) cudaFree(p);
        for (int l = 0; l <= kMaxLayers; l++) {
            cudaFree(bufs.A[l]);
            cudaFree(bufs.dZ[l]);
        }
        drop_predict();
        cudaFree(lossp);
        cudaFree(loss);
        if (own_stream && stream) cudaStreamDestroy(stream);
    }
};

namespace {

void merr(lbs_mlp *n, const char *fmt, ...) {
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(n->err, sizeof(n->err), fmt, ap);
    va_end(ap);
}

#define MCK(call)                                                                         \
    do {                                                                                  \
        cudaError_t e_ = (call);                                                          \
        if (e_ != cudaSuccess) {                                                          \
            merr(net, "%s failed: %s (%s:%d)", #call, cudaGetErrorString(e_), __FILE__,   \
                 __LINE__);                                                               \
            return LBS_ECUDA;                                                             \
        }                                                                                 \
    } while (0)

template <int ROWS>
size_t forward_smem(const Shape &s) {
    using T = Tile<ROWS>;
    return ((size_t)s.wmax + kMaxWidth * T::RS + kNarrow * T::NT) * sizeof(float);
}
size_t pass_smem(const Shape &s) { return pass_floats(s) * sizeof(float); }

// the copy of the weights that a kernel about to be queued multiplies by
int ensure_weights(lbs_mlp *net, bool bf16) {
    bool &valid = bf16 ? net->bf_valid : net->w_valid;
    if (valid) return LBS_OK;
    const long long n = (long long)net->E * net->s.P;
    const int g = (int)std::min<long long>((n + 255) / 256, 4096);
    if (bf16)
        k_copy_weights<true><<<g, 256, 0, net->stream>>>(net->params, net->s, net->E, net->Wbf);
    else
        k_copy_weights<false><<<g, 256, 0, net->stream>>>(net->params, net->s, net->E, net->W);
    MCK(cudaGetLastError());
    valid = true;
    return LBS_OK;
}

// outputs y [E][B][n_out] of the rows x (xstride between members; 0: the same
// rows for every member).  64 rows a block when that fills the chip (5 x 1024
// rows on 152 SMs do not: 80 blocks), else 16: 4 times the blocks, each a
// quarter of the work.
int forward(lbs_mlp *net, const float *x, long long xstride, int B, bool bf16, float *y) {
    int r = ensure_weights(net, bf16);
    if (r) return r;
    const Shape &s = net->s;
    const float *W = bf16 ? net->Wbf : net->W;
    const long long wide = (long long)((B + 63) / 64) * net->E;
    if (wide >= net->sms)
        k_net_forward<64><<<dim3((B + 63) / 64, net->E), Tile<64>::NT, forward_smem<64>(s),
                            net->stream>>>(W, s, x, xstride, B, y);
    else
        k_net_forward<16><<<dim3((B + 15) / 16, net->E), Tile<16>::NT, forward_smem<16>(s),
                            net->stream>>>(W, s, x, xstride, B, y);
    MCK(cudaGetLastError());
    return LBS_OK;
}

int pass_tiles(int B) { return (B + kTrainRows - 1) / kTrainRows; }

// activations, loss and gradient of every member for its minibatch (ndata > 0:
// drawn from the data set, else the rows X, Y [E][B][.]); ad.on: Adam's step
int pass(lbs_mlp *net, const float *X, const float *Y, int ndata, int B, unsigned long long seed,
         const Adam &ad) {
    int r = ensure_weights(net, false);
    if (r) return r;
    const Shape &s = net->s;
    k_net_pass<<<dim3(pass_tiles(B), net->E), Tile<kTrainRows>::NT, pass_smem(s), net->stream>>>(
        net->W, s, X, Y, ndata, B, seed, net->t, net->bufs, net->lossp);
    int tiles = 0;
    for (int l = 1; l <= s.L; l++)
        tiles += ((s.d[l - 1] + kUpTile - 1) / kUpTile) * ((s.d[l] + kUpTile - 1) / kUpTile);
    k_net_update<<<dim3(tiles, net->E), 256, 0, net->stream>>>(
        s, B, net->bufs, ad, net->params, net->grad, net->m, net->v, net->W);
    MCK(cudaGetLastError());
    return LBS_OK;
}

int sum_loss(lbs_mlp *net, int B) {
    k_loss_sum<<<net->E, 32, 0, net->stream>>>(net->lossp, pass_tiles(B),
                                               (long long)B * net->s.d[net->s.L], net->loss);
    MCK(cudaGetLastError());
    return LBS_OK;
}

// the constants of the next Adam step, counted
Adam next_adam(lbs_mlp *net, float lr, float b1, float b2, float eps) {
    net->t += 1;
    Adam a;
    a.on = 1;
    a.lr = lr;
    a.b1 = b1;
    a.b2 = b2;
    a.eps = eps;
    a.c1 = float(1.0 - std::pow(double(b1), double(net->t)));
    a.c2 = float(1.0 - std::pow(double(b2), double(net->t)));
    return a;
}

}  // namespace

extern "C" {

int lbs_mlp_create(int members, int n_in, int width, int depth, int n_out, int max_batch,
                   void *stream, lbs_mlp **out) {
    if (!out) return LBS_EINVAL;
    lbs_mlp *net = new (std::nothrow) lbs_mlp();
    *out = net;
    if (!net) return LBS_ENOMEM;
    if (members < 1 || n_in < 1 || n_out < 1 || width < 1 || depth < 1 || max_batch < 1 ||
        n_in > kMaxWidth || width > kMaxWidth || n_out > kMaxWidth || depth + 1 > kMaxLayers) {
        merr(net, "network %d -> %d x %d -> %d (E = %d, batch %d): widths 1..%d, depth 1..%d",
             n_in, width, depth, n_out, members, max_batch, kMaxWidth, kMaxLayers - 1);
        return LBS_EINVAL;
    }
    net->E = members;
    net->B = max_batch;
    Shape &s = net->s;
    s.L = depth + 1;
    s.d[0] = n_in;
    for (int l = 1; l <= depth; l++) s.d[l] = width;
    s.d[s.L] = n_out;
    long long off = 0;
    s.S = 0;
    s.wmax = 0;
    for (int l = 0; l <= s.L; l++) s.ld[l] = up4(s.d[l]);
    for (int l = 1; l <= s.L; l++) {
        s.woff[l] = off;
        off += (long long)s.d[l] * s.d[l - 1];
        s.boff[l] = off;
        off += s.d[l];
        const int nt = s.d[l - 1] * s.ld[l], nn = s.d[l] * s.ld[l - 1];
        s.wt[l] = s.S;
        s.wn[l] = s.wt[l] + nt;
        s.bs[l] = s.wn[l] + nn;
        s.S = s.bs[l] + s.ld[l];
        s.wmax = std::max(s.wmax, std::max(nt, nn));
    }
    s.P = off;
    if (stream) {
        net->stream = (cudaStream_t)stream;
    } else {
        MCK(cudaStreamCreateWithFlags(&net->stream, cudaStreamNonBlocking));
        net->own_stream = true;
    }
    int dev = 0;
    MCK(cudaGetDevice(&dev));
    MCK(cudaDeviceGetAttribute(&net->sms, cudaDevAttrMultiProcessorCount, dev));
    // (the largest shapes, so that no network lowers what another one needs)
    const int kMaxSmem = 227 * 1024 - 1024;
    MCK(cudaFuncSetAttribute(k_net_forward<64>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             112 * 1024));
    MCK(cudaFuncSetAttribute(k_net_forward<16>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             112 * 1024));
    MCK(cudaFuncSetAttribute(k_net_pass, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem));
    const long long EP = (long long)members * s.P, ES = (long long)members * s.S;
    MCK(cudaMalloc(&net->params, EP * sizeof(float)));
    MCK(cudaMalloc(&net->grad, EP * sizeof(float)));
    MCK(cudaMalloc(&net->m, EP * sizeof(float)));
    MCK(cudaMalloc(&net->v, EP * sizeof(float)));
    MCK(cudaMalloc(&net->W, ES * sizeof(float)));
    MCK(cudaMalloc(&net->Wbf, ES * sizeof(float)));
    MCK(cudaMemset(net->m, 0, EP * sizeof(float)));
    MCK(cudaMemset(net->v, 0, EP * sizeof(float)));
    MCK(cudaMemset(net->params, 0, EP * sizeof(float)));
    MCK(cudaMemset(net->W, 0, ES * sizeof(float)));
    MCK(cudaMemset(net->Wbf, 0, ES * sizeof(float)));
    const long long EB = (long long)members * max_batch;
    for (int l = 0; l < s.L; l++) {
        MCK(cudaMalloc(&net->bufs.A[l], EB * s.ld[l] * sizeof(float)));
        MCK(cudaMalloc(&net->bufs.dZ[l + 1], EB * s.ld[l + 1] * sizeof(float)));
    }
    MCK(cudaMalloc(&net->x, EB * n_in * sizeof(float)));
    MCK(cudaMalloc(&net->y, EB * n_out * sizeof(float)));
    MCK(cudaMalloc(&net->T, EB * n_out * sizeof(float)));
    MCK(cudaMalloc(&net->stats, 2 * (long long)max_batch * n_out * sizeof(float)));
    MCK(cudaMalloc(&net->lossp, (long long)members * pass_tiles(max_batch) * sizeof(double)));
    MCK(cudaMalloc(&net->loss, members * sizeof(double)));
    MCK(cudaStreamSynchronize(0));  // (the clears above, before work on the network's stream)
    return LBS_OK;
}

int lbs_mlp_param_count(const lbs_mlp *net) { return net ? (int)net->s.P : 0; }

int lbs_mlp_init(lbs_mlp *net, unsigned long long seed) {
    if (!net) return LBS_EINVAL;
    const Shape &s = net->s;
    long long *dw = nullptr;
    int *dd = nullptr;
    MCK(cudaMalloc(&dw, 2 * (kMaxLayers + 1) * sizeof(long long)));
    MCK(cudaMalloc(&dd, (kMaxLayers + 1) * sizeof(int)));
    MCK(cudaMemcpyAsync(dw, s.woff, (kMaxLayers + 1) * sizeof(long long), cudaMemcpyHostToDevice, net->stream));
    MCK(cudaMemcpyAsync(dw + kMaxLayers + 1, s.boff, (kMaxLayers + 1) * sizeof(long long),
                        cudaMemcpyHostToDevice, net->stream));
    MCK(cudaMemcpyAsync(dd, s.d, (kMaxLayers + 1) * sizeof(int), cudaMemcpyHostToDevice, net->stream));
    const long long n = (long long)net->E * s.P;
    k_init<<<(int)std::min<long long>((n + 255) / 256, 4096), 256, 0, net->stream>>>(
        net->params, n, dw, dw + kMaxLayers + 1, dd, s.L, s.P, seed);
    MCK(cudaGetLastError());
    MCK(cudaStreamSynchronize(net->stream));
    cudaFree(dw);
    cudaFree(dd);
    MCK(cudaMemsetAsync(net->m, 0, n * sizeof(float), net->stream));
    MCK(cudaMemsetAsync(net->v, 0, n * sizeof(float), net->stream));
    net->t = 0;
    net->w_valid = net->bf_valid = false;
    return LBS_OK;
}

int lbs_mlp_set_params(lbs_mlp *net, const float *host) {
    if (!net || !host) return LBS_EINVAL;
    net->w_valid = net->bf_valid = false;
    MCK(cudaMemcpyAsync(net->params, host, (long long)net->E * net->s.P * sizeof(float),
                        cudaMemcpyHostToDevice, net->stream));
    MCK(cudaStreamSynchronize(net->stream));
    return LBS_OK;
}

int lbs_mlp_get_params(lbs_mlp *net, float *host) {
    if (!net || !host) return LBS_EINVAL;
    MCK(cudaMemcpyAsync(host, net->params, (long long)net->E * net->s.P * sizeof(float),
                        cudaMemcpyDeviceToHost, net->stream));
    MCK(cudaStreamSynchronize(net->stream));
    return LBS_OK;
}

int lbs_mlp_forward(lbs_mlp *net, const float *x, int batch, int bf16, float *y) {
    if (!net || !x || !y || batch < 1 || batch > net->B) return LBS_EINVAL;
    const Shape &s = net->s;
    MCK(cudaMemcpyAsync(net->x, x, (long long)net->E * batch * s.d[0] * sizeof(float),
                        cudaMemcpyHostToDevice, net->stream));
    int r = forward(net, net->x, (long long)batch * s.d[0], batch, bf16 != 0, net->y);
    if (r) return r;
    MCK(cudaMemcpyAsync(y, net->y, (long long)net->E * batch * s.d[s.L] * sizeof(float),
                        cudaMemcpyDeviceToHost, net->stream));
    MCK(cudaStreamSynchronize(net->stream));
    return LBS_OK;
}

int lbs_mlp_gradient(lbs_mlp *net, const float *x, const float *t, int batch, float *grad,
                     double *loss) {
    if (!net || !x || !t || batch < 1 || batch > net->B) return LBS_EINVAL;
    const Shape &s = net->s;
    MCK(cudaMemcpyAsync(net->x, x, (long long)net->E * batch * s.d[0] * sizeof(float),
                        cudaMemcpyHostToDevice, net->stream));
    MCK(cudaMemcpyAsync(net->T, t, (long long)net->E * batch * s.d[s.L] * sizeof(float),
                        cudaMemcpyHostToDevice, net->stream));
    Adam off = {};
    int r = pass(net, net->x, net->T, 0, batch, 0, off);
    if (!r) r = sum_loss(net, batch);
    if (r) return r;
    if (grad)
        MCK(cudaMemcpyAsync(grad, net->grad, (long long)net->E * s.P * sizeof(float),
                            cudaMemcpyDeviceToHost, net->stream));
    if (loss)
        MCK(cudaMemcpyAsync(loss, net->loss, net->E * sizeof(double), cudaMemcpyDeviceToHost,
                            net->stream));
    MCK(cudaStreamSynchronize(net->stream));
    return LBS_OK;
}

int lbs_mlp_set_grad(lbs_mlp *net, const float *host) {
    if (!net || !host) return LBS_EINVAL;
    MCK(cudaMemcpyAsync(net->grad, host, (long long)net->E * net->s.P * sizeof(float),
                        cudaMemcpyHostToDevice, net->stream));
    MCK(cudaStreamSynchronize(net->stream));
    return LBS_OK;
}

int lbs_mlp_adam_step(lbs_mlp *net, float lr, float beta1, float beta2, float eps) {
    if (!net || !(lr >= 0) || !(beta1 >= 0 && beta1 < 1) || !(beta2 >= 0 && beta2 < 1) ||
        !(eps > 0))
        return LBS_EINVAL;
    const Adam a = next_adam(net, lr, beta1, beta2, eps);
    const long long n = (long long)net->E * net->s.P;
    net->w_valid = net->bf_valid = false;
    k_adam<<<(int)std::min<long long>((n + 255) / 256, 4096), 256, 0, net->stream>>>(
        net->params, net->grad, net->m, net->v, n, a);
    MCK(cudaGetLastError());
    MCK(cudaStreamSynchronize(net->stream));
    return LBS_OK;
}

int lbs_mlp_set_data(lbs_mlp *net, const float *X, const float *Y, int n) {
    if (!net || !X || !Y || n < 1) return LBS_EINVAL;
    cudaFree(net->X);
    cudaFree(net->Yd);
    net->X = net->Yd = nullptr;
    MCK(cudaMalloc(&net->X, (long long)n * net->s.d[0] * sizeof(float)));
    MCK(cudaMalloc(&net->Yd, (long long)n * net->s.d[net->s.L] * sizeof(float)));
    MCK(cudaMemcpyAsync(net->X, X, (long long)n * net->s.d[0] * sizeof(float),
                        cudaMemcpyHostToDevice, net->stream));
    MCK(cudaMemcpyAsync(net->Yd, Y, (long long)n * net->s.d[net->s.L] * sizeof(float),
                        cudaMemcpyHostToDevice, net->stream));
    MCK(cudaStreamSynchronize(net->stream));
    net->ndata = n;
    return LBS_OK;
}

int lbs_mlp_train(lbs_mlp *net, int iters, int batch, float lr, float beta1, float beta2,
                  float eps, unsigned long long seed, double *loss) {
    if (!net || iters < 0 || batch < 1 || batch > net->B || !net->X) return LBS_EINVAL;
    for (int it = 0; it < iters; it++) {
        net->bf_valid = false;
        // (the rows are drawn by the number of steps taken before this one)
        const long long t0 = net->t;
        const Adam a = next_adam(net, lr, beta1, beta2, eps);
        net->t = t0;
        int r = pass(net, net->X, net->Yd, net->ndata, batch, seed, a);
        if (r) return r;
        net->t = t0 + 1;
    }
    if (iters > 0) {
        int r = sum_loss(net, batch);
        if (r) return r;
    }
    if (loss)
        MCK(cudaMemcpyAsync(loss, net->loss, net->E * sizeof(double), cudaMemcpyDeviceToHost,
                            net->stream));
    MCK(cudaStreamSynchronize(net->stream));
    return LBS_OK;
}

// rows a chunk of predict takes: up to 65,536 and a workspace of 64 MiB of
// outputs, kept for the next call, where n exceeds max_batch; without that
// memory chunks of max_batch rows in the buffers that are there
static int predict_rows(lbs_mlp *net, int n) {
    if (n <= net->B) return net->B;
    const Shape &s = net->s;
    const int nin = s.d[0], nout = s.d[s.L];
    const long long cap = std::max<long long>(1, (16ll << 20) / ((long long)net->E * nout));
    const int rows = (int)std::min<long long>(std::min<long long>(n, 65536), cap);
    if (rows <= net->B) return net->B;
    if (rows <= net->prows) return net->prows;
    cudaStreamSynchronize(net->stream);
    net->drop_predict();
    if (cudaMalloc(&net->px, (long long)rows * nin * sizeof(float)) != cudaSuccess ||
        cudaMalloc(&net->py, (long long)net->E * rows * nout * sizeof(float)) != cudaSuccess ||
        cudaMalloc(&net->pstats, 2 * (long long)rows * nout * sizeof(float)) != cudaSuccess) {
        cudaGetLastError();
        net->drop_predict();
        return net->B;
    }
    net->prows = rows;
    return rows;
}

int lbs_mlp_predict(lbs_mlp *net, const float *x, int n, int bf16, float *mean, float *sd) {
    if (!net || !x || !mean || !sd || n < 1) return LBS_EINVAL;
    const Shape &s = net->s;
    const int nin = s.d[0], nout = s.d[s.L];
    const int rows = predict_rows(net, n);
    const bool big = rows > net->B;
    float *xd = big ? net->px : net->x, *yd = big ? net->py : net->y;
    float *st = big ? net->pstats : net->stats;
    for (int q0 = 0; q0 < n; q0 += rows) {
        const int m = std::min(rows, n - q0);
        MCK(cudaMemcpyAsync(xd, x + (long long)q0 * nin, (long long)m * nin * sizeof(float),
                            cudaMemcpyHostToDevice, net->stream));
        int r = forward(net, xd, 0, m, bf16 != 0, yd);
        if (r) return r;
        const long long cnt = (long long)m * nout;
        k_stats<<<(int)((cnt + 255) / 256), 256, 0, net->stream>>>(yd, net->E, cnt, st, st + cnt);
        MCK(cudaGetLastError());
        MCK(cudaMemcpyAsync(mean + (long long)q0 * nout, st, cnt * sizeof(float),
                            cudaMemcpyDeviceToHost, net->stream));
        MCK(cudaMemcpyAsync(sd + (long long)q0 * nout, st + cnt, cnt * sizeof(float),
                            cudaMemcpyDeviceToHost, net->stream));
        MCK(cudaStreamSynchronize(net->stream));
    }
    return LBS_OK;
}

void lbs_mlp_destroy(lbs_mlp *net) { delete net; }

const char *lbs_mlp_last_error(const lbs_mlp *net) {
    if (!net) return "null network";
    return net->err[0] ? net->err : "no error";
}

}  // extern "C"
