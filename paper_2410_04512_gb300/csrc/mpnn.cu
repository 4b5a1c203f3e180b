// mpnn.cu -- learned warm start: a message-passing network over the
// collision graph that predicts the PCG initial guess v0 (the paper has no
// learned component; the solver's own iterations measure the prediction).
//
// Network (width 64, 3 message-passing layers, BF16 weights, FP32
// activations and accumulation):
//   basis  b0 = D^-1 F (block Jacobi), b1 = P^-1 F (spanning forest),
//          b2 = previous velocity (or 0)
//   x_i    = (|b0|, |b1|, |b2|, b0.b1, b0.b2, b1.b2) / (mean |b1|)^(1|2),
//            deg_i / 6, 1
//   h0     = relu(W_in x + b_in)
//   h_l+1  = relu(W_l [h_l ; mean_{j~i} h_l,j] + c_l),   l = 0, 1, 2
//   c      = W_out h3 + b_out,   v0_i = sum_k c_ik b_i^(k)
// Every feature is rotation invariant and v0 is a scalar mix of equivariant
// fields, so the prediction rotates with the configuration.
//
// Training (online, on solutions of earlier steps): loss
// |v0 - v*|^2 / |v*|^2, hand-written backward kernels, Adam on FP32 master
// weights, BF16 copies refreshed after every step.  Weight gradients are
// reduced per block and then in block order (deterministic).
#include <cuda_bf16.h>

#include <cfloat>

#include "sgp_internal.cuh"

sgp_status spmv64(sgp_ctx *ctx, const sgp_matrix *M, const double *v, double *y);

namespace {

constexpr int H = 64, KB = 3, DIN = 8, H2 = 2 * H;
// parameter layout (FP32 master, flat): W_in, b_in, {W_l, c_l} x 3, W_out, b_out
constexpr int OFF_WIN = 0, OFF_BIN = OFF_WIN + H * DIN;
constexpr int OFF_L0 = OFF_BIN + H;
constexpr int LAYER = H * H2 + H;
constexpr int OFF_WOUT = OFF_L0 + 3 * LAYER, OFF_BOUT = OFF_WOUT + KB * H;
constexpr int NPARAM = OFF_BOUT + KB;
static_assert(NPARAM == SGP_MPNN_PARAMS, "parameter layout");
constexpr int TB = 256;          // threads per block
constexpr int CHUNK = 256;       // nodes per block in the weight-gradient reductions

__device__ __forceinline__ float bf(const __nv_bfloat16 *w, int k) { return __bfloat162float(w[k]); }

// ---------------------------------------------------------------- features
// b0 = D^-1 F with the block-Jacobi inverse (sym6 per row)
__global__ void k_mp_jacobi(int64_t n, const double *__restrict__ jac, const double *__restrict__ F, double *b0)
{
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) sym_mv(jac + 6 * i, F + 3 * i, b0 + 3 * i);
}

// The mean of |b1_i| and the scale 1 / mean (1 if it vanishes): blocks, then
// the last block (fixed order).
__global__ void k_mp_norm_sum(int64_t n, const double *__restrict__ b1, double *partials, unsigned *counter,
                              double *out)
{
    __shared__ double sh[TB / 32];
    double s = 0.0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        s += sqrt(b1[3 * i] * b1[3 * i] + b1[3 * i + 1] * b1[3 * i + 1] + b1[3 * i + 2] * b1[3 * i + 2]);
    s = block_sum<TB>(s, sh);
    if (threadIdx.x == 0) partials[blockIdx.x] = s;
    if (last_block(counter)) {
        double t = sum_partials<TB>(partials, gridDim.x, sh);
        if (threadIdx.x == 0) {
            const double mean = t / (double)(n > 0 ? n : 1);
            out[0] = mean;
            out[1] = fmin(1.0 / (mean > 0.0 ? mean : 1.0), DBL_MAX);
        }
    }
}

// FP64 bound: the scale comes as a reciprocal, as a division is some ten
// instructions (seven of them per cell: 26 us at 1e5 cells, 15 so).  Twice in
// turn, not as a square, which leaves the range of doubles at 1e154.
__global__ void k_mp_features(int64_t n, const double *__restrict__ b0, const double *__restrict__ b1,
                              const double *__restrict__ b2, const int32_t *__restrict__ row_ptr,
                              const double *__restrict__ mean_b1, float *x)
{
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double s = mean_b1[1];
    const double *a = b0 + 3 * i, *b = b1 + 3 * i, *c = b2 + 3 * i;
    auto dot = [](const double *u, const double *v) { return u[0] * v[0] + u[1] * v[1] + u[2] * v[2]; };
    float *o = x + DIN * i;
    o[0] = (float)(sqrt(dot(a, a)) * s);
    o[1] = (float)(sqrt(dot(b, b)) * s);
    o[2] = (float)(sqrt(dot(c, c)) * s);
    o[3] = (float)(dot(a, b) * s * s);
    o[4] = (float)(dot(a, c) * s * s);
    o[5] = (float)(dot(b, c) * s * s);
    o[6] = (float)((row_ptr[i + 1] - row_ptr[i]) * (1.0 / 6.0));
    o[7] = 1.0f;
}

// ------------------------------------------------------------ dense layers
// Y (n x DOUT) = act(X Wt + bias) where X = [X1 (n x D1), X2 (n x D2)] and the
// BF16 matrix W is DOUT x (D1 + D2), or, TRANS, Y = X W with W of shape
// (D1 + D2) x DOUT (the backward product dX = dZ W; the second half of the
// outputs, dA, is scaled by 1 / deg of its row for the transposed mean).
// FP32 FMAs on register tiles: a block holds the weights (FP32, [k][o]) and a
// tile of 16 NU nodes' inputs (row-major, padded) in shared memory; a thread
// computes NU nodes (ty, ty + 16, ...) x 4 or 8 outputs, reading 16 bytes per
// load: with NU = 8 a warp takes 16 to 24 shared-memory wavefronts per 128 to
// 256 FMAs, so the FMA pipe is the bound.  Weights are read 16 bytes at a time
// (8 inputs of one output) and spread over the rows without bank conflicts.
// Each output accumulates bias + sum_k x_k w_k in ascending k.  1e5 cells:
// forward layer 80 -> 69 us, backward product 147 -> 53 us.
template <int D1, int D2, int DOUT, bool TRANS, bool RELU, int NU>
__global__ void __launch_bounds__(TB, 2) k_mp_dense(int64_t n, const float *__restrict__ X1, const float *__restrict__ X2,
                                                    const __nv_bfloat16 *__restrict__ W,
                                                    const __nv_bfloat16 *__restrict__ bias,
                                                    const int32_t *__restrict__ row_ptr, float *__restrict__ Y)
{
    constexpr int DI = D1 + D2, XP = DI + 4, OG = DOUT / 64, DN = 16 * NU;
    static_assert(DI % 8 == 0 && D1 % 4 == 0 && (DOUT == 64 || DOUT == 128), "tile shape");
    extern __shared__ __align__(16) float dsm[];
    float *wt = dsm;                    // [DI][DOUT]
    float *xs = dsm + DI * DOUT;        // [DN][XP]
    for (int c = threadIdx.x; c < DI * DOUT / 8; c += TB) {
        if (TRANS) {
            const int t = 8 * c;        // row k, outputs o..o+7
            const uint4 q = *reinterpret_cast<const uint4 *>(W + t);
            const uint32_t u[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                wt[t + 2 * j] = __uint_as_float(u[j] << 16);
                wt[t + 2 * j + 1] = __uint_as_float(u[j] & 0xffff0000u);
            }
        } else {
            const int o = c % DOUT, k = 8 * (c / DOUT);
            const uint4 q = *reinterpret_cast<const uint4 *>(W + o * DI + k);
            const uint32_t u[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                wt[(k + 2 * j) * DOUT + o] = __uint_as_float(u[j] << 16);
                wt[(k + 2 * j + 1) * DOUT + o] = __uint_as_float(u[j] & 0xffff0000u);
            }
        }
    }
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    float bv[4 * OG];
#pragma unroll
    for (int v = 0; v < 4 * OG; ++v) bv[v] = bias ? bf(bias, (v >> 2) * 64 + 4 * tx + (v & 3)) : 0.f;
    const int64_t ntiles = (n + DN - 1) / DN;
    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int64_t base = tile * DN;
        __syncthreads();
#pragma unroll 8
        for (int c = threadIdx.x; c < DN * (DI / 4); c += TB) {
            const int node = c / (DI / 4), k = 4 * (c % (DI / 4));
            const int64_t i = base + node;
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (i < n) v = k < D1 ? *reinterpret_cast<const float4 *>(X1 + i * D1 + k)
                                  : *reinterpret_cast<const float4 *>(X2 + i * D2 + (k - D1));
            *reinterpret_cast<float4 *>(xs + node * XP + k) = v;
        }
        __syncthreads();
        float acc[NU][4 * OG];
#pragma unroll
        for (int u = 0; u < NU; ++u)
#pragma unroll
            for (int v = 0; v < 4 * OG; ++v) acc[u][v] = bv[v];
#pragma unroll 1
        for (int k = 0; k < DI; k += 4) {
            float4 xv[NU];
#pragma unroll
            for (int u = 0; u < NU; ++u) xv[u] = *reinterpret_cast<const float4 *>(xs + (ty + 16 * u) * XP + k);
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)
#pragma unroll
                for (int g = 0; g < OG; ++g) {
                    const float4 wv = *reinterpret_cast<const float4 *>(wt + (k + kk) * DOUT + 64 * g + 4 * tx);
#pragma unroll
                    for (int u = 0; u < NU; ++u) {
                        const float xk = kk == 0 ? xv[u].x : kk == 1 ? xv[u].y : kk == 2 ? xv[u].z : xv[u].w;
                        acc[u][4 * g] = fmaf(xk, wv.x, acc[u][4 * g]);
                        acc[u][4 * g + 1] = fmaf(xk, wv.y, acc[u][4 * g + 1]);
                        acc[u][4 * g + 2] = fmaf(xk, wv.z, acc[u][4 * g + 2]);
                        acc[u][4 * g + 3] = fmaf(xk, wv.w, acc[u][4 * g + 3]);
                    }
                }
        }
#pragma unroll
        for (int u = 0; u < NU; ++u) {
            const int64_t i = base + ty + 16 * u;
            if (i >= n) continue;
#pragma unroll
            for (int g = 0; g < OG; ++g) {
                float4 o4 = make_float4(acc[u][4 * g], acc[u][4 * g + 1], acc[u][4 * g + 2], acc[u][4 * g + 3]);
                if (RELU) o4 = make_float4(fmaxf(o4.x, 0.f), fmaxf(o4.y, 0.f), fmaxf(o4.z, 0.f), fmaxf(o4.w, 0.f));
                if (TRANS && g == 1) {
                    const float inv = 1.0f / (float)max(row_ptr[i + 1] - row_ptr[i], 1);
                    o4 = make_float4(o4.x * inv, o4.y * inv, o4.z * inv, o4.w * inv);
                }
                *reinterpret_cast<float4 *>(Y + i * DOUT + 64 * g + 4 * tx) = o4;
            }
        }
    }
}

// The sum of the neighbours' rows (16 lanes per node, 16 bytes per lane; the
// neighbours' indices in one load, their rows four at a time), in ascending
// column order.
__device__ __forceinline__ void row_sum(const int32_t *__restrict__ col, int32_t s0, int32_t s1,
                                        const float *__restrict__ X, int pitch, float4 &a)
{
    const int lane = threadIdx.x & 31, l = lane & 15;
    const unsigned mask = 0xffffu << (lane & 16);
    for (int32_t b = s0; b < s1; b += 16) {
        const int cnt = min(16, s1 - b);
        const int32_t c = l < cnt ? col[b + l] : 0;
        for (int j = 0; j < cnt; j += 4) {
            float4 v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int32_t i = __shfl_sync(mask, c, (lane & 16) | min(j + u, 15));
                v[u] = j + u < cnt ? reinterpret_cast<const float4 *>(X + (int64_t)i * pitch)[l]
                                   : make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                a.x += v[u].x; a.y += v[u].y; a.z += v[u].z; a.w += v[u].w;
            }
        }
    }
}

// A_i = mean_{j ~ i} H_j (0 for an isolated cell).
__global__ void __launch_bounds__(TB) k_mp_agg(int64_t n, const int32_t *__restrict__ row_ptr,
                                               const int32_t *__restrict__ col, const float *__restrict__ Hm, float *A)
{
    const int64_t w = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 4;
    if (w >= n) return;
    const int32_t s0 = row_ptr[w], s1 = row_ptr[w + 1];
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
    row_sum(col, s0, s1, Hm, H, a);
    const float inv = 1.0f / (float)max(s1 - s0, 1);
    reinterpret_cast<float4 *>(A + w * H)[threadIdx.x & 15] = make_float4(a.x * inv, a.y * inv, a.z * inv, a.w * inv);
}

__device__ __forceinline__ float4 relu_mask(float4 y, float4 d)
{
    return make_float4(y.x > 0.f ? d.x : 0.f, y.y > 0.f ? d.y : 0.f, y.z > 0.f ? d.z : 0.f, y.w > 0.f ? d.w : 0.f);
}

// Transpose of the mean, dH_j = dSelf_j + sum_{i ~ j} dA_i / deg_i (dA comes
// scaled), through the ReLU of H: dZ_j = dH_j where H_j > 0.
__global__ void __launch_bounds__(TB) k_mp_agg_t(int64_t n, const int32_t *__restrict__ row_ptr,
                                                 const int32_t *__restrict__ col, const float *__restrict__ dU,
                                                 const float *__restrict__ Hm, float *dZ)
{
    const int64_t w = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 4;
    if (w >= n) return;
    const int l = threadIdx.x & 15;
    float4 a = reinterpret_cast<const float4 *>(dU + w * H2)[l];
    const float4 y = reinterpret_cast<const float4 *>(Hm + w * H)[l];
    row_sum(col, row_ptr[w], row_ptr[w + 1], dU + H, H2, a);
    reinterpret_cast<float4 *>(dZ + w * H)[l] = relu_mask(y, a);
}

// The output layer backwards: dZ = (W_out^T dc) where H > 0.
__global__ void __launch_bounds__(TB) k_mp_out_t(int64_t n, const float *__restrict__ dc,
                                                 const __nv_bfloat16 *__restrict__ W, const float *__restrict__ Hm, float *dZ)
{
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, i = t >> 4;
    if (i >= n) return;
    const int l = (int)(t & 15);
    float a[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int k = 0; k < KB; ++k) {
        const float d = dc[i * KB + k];
#pragma unroll
        for (int v = 0; v < 4; ++v) a[v] = fmaf(d, bf(W, k * H + 4 * l + v), a[v]);
    }
    reinterpret_cast<float4 *>(dZ)[t] = relu_mask(reinterpret_cast<const float4 *>(Hm)[t], make_float4(a[0], a[1], a[2], a[3]));
}

// c = W_out h3 + b_out (kept), v0 = sum_k c_k b^(k) in FP64.  16 lanes per node
// for c, four nodes each; then a lane per component of v0, so that the FP64
// instructions run on full warps (with three of 16 lanes: 22 us at 1e5
// cells).
constexpr int ON = 64;   // nodes per block
__global__ void __launch_bounds__(TB) k_mp_out(int64_t n, const float *__restrict__ h3, const __nv_bfloat16 *__restrict__ Wout,
                                               const __nv_bfloat16 *__restrict__ bout, const double *__restrict__ b0,
                                               const double *__restrict__ b1, const double *__restrict__ b2, float *c,
                                               double *v0)
{
    __shared__ float cs[ON * KB];
    const int64_t base = blockIdx.x * (int64_t)ON;
    const int l = threadIdx.x & 15, node = threadIdx.x >> 4;
    const int nn = (int)min((int64_t)ON, n - base);
    float w[KB][4], bk[KB];
#pragma unroll
    for (int k = 0; k < KB; ++k) {
        bk[k] = bf(bout, k);
#pragma unroll
        for (int v = 0; v < 4; ++v) w[k][v] = bf(Wout, k * H + 4 * l + v);
    }
    float4 h[ON / 16];
#pragma unroll
    for (int u = 0; u < ON / 16; ++u)
        h[u] = node + 16 * u < nn ? reinterpret_cast<const float4 *>(h3 + (base + node + 16 * u) * H)[l]
                                  : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int u = 0; u < ON / 16; ++u) {
        float ck[KB];
#pragma unroll
        for (int k = 0; k < KB; ++k) {
            ck[k] = fmaf(h[u].x, w[k][0], fmaf(h[u].y, w[k][1], fmaf(h[u].z, w[k][2], h[u].w * w[k][3])));
#pragma unroll
            for (int b = 8; b > 0; b >>= 1) ck[k] += __shfl_xor_sync(0xffffffffu, ck[k], b);
            ck[k] += bk[k];
        }
        if (l < KB) cs[(node + 16 * u) * KB + l] = l == 0 ? ck[0] : l == 1 ? ck[1] : ck[2];
    }
    __syncthreads();
    if (threadIdx.x >= 3 * nn) return;
    const float *q = cs + threadIdx.x / 3 * KB;
    const int64_t at = 3 * base + threadIdx.x;
    c[at] = cs[threadIdx.x];
    v0[at] = (double)q[0] * b0[at] + (double)q[1] * b1[at] + (double)q[2] * b2[at];
}

// out[0] = x . y, out[1] = z . w over 3n values (blocks, then the last
// block in a fixed order)
__global__ void k_mp_dot2(int64_t n3, const double *__restrict__ x, const double *__restrict__ y,
                          const double *__restrict__ z, const double *__restrict__ w, double *partials,
                          unsigned *counter, double *out)
{
    __shared__ double sh[TB / 32];
    double e = 0.0, t = 0.0;
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n3; k += (int64_t)gridDim.x * blockDim.x) {
        e = fma(x[k], y[k], e);
        t = fma(z[k], w[k], t);
    }
    double a = block_sum<TB>(e, sh);
    if (threadIdx.x == 0) partials[2 * blockIdx.x] = a;
    double b = block_sum<TB>(t, sh);
    if (threadIdx.x == 0) partials[2 * blockIdx.x + 1] = b;
    if (last_block(counter)) {
        double A = 0.0, B = 0.0;
        for (unsigned k = threadIdx.x; k < gridDim.x; k += TB) {
            A += __ldcg(partials + 2 * k);
            B += __ldcg(partials + 2 * k + 1);
        }
        A = block_sum<TB>(A, sh);
        B = block_sum<TB>(B, sh);
        if (threadIdx.x == 0) {
            out[0] = A;
            out[1] = B;
        }
    }
}

__global__ void k_mp_diff(int64_t n3, const double *__restrict__ a, const double *__restrict__ b, double *e)
{
    int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (k < n3) e[k] = a[k] - b[k];
}

// dc_ik = dv_i . b^(k)_i with dv = 2 g / nd[1] (g = v0 - v* for the l2
// loss, Gamma (v0 - v*) for the energy loss; nd[1] the normaliser)
__global__ void k_mp_dc(int64_t n, const double *__restrict__ g, const double *__restrict__ b0,
                        const double *__restrict__ b1, const double *__restrict__ b2, const double *__restrict__ nd,
                        float *dc)
{
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double s = nd[1] > 0 ? 2.0 / nd[1] : 0.0;
    double dv[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) dv[d] = s * g[3 * i + d];
    const double *bb[3] = {b0, b1, b2};
#pragma unroll
    for (int k = 0; k < KB; ++k)
        dc[i * KB + k] = (float)(dv[0] * bb[k][3 * i] + dv[1] * bb[k][3 * i + 1] + dv[2] * bb[k][3 * i + 2]);
}

// L = nd[0] / nd[1]
__global__ void k_mp_ratio(const double *__restrict__ nd, double *L)
{
    if (threadIdx.x == 0) L[0] = nd[1] > 0 ? nd[0] / nd[1] : 0.0;
}

// v0 *= alpha with alpha = nd[0] / nd[1] (the minimal-residual step), kept
// as is when the denominator vanishes or alpha is not finite
__global__ void k_mp_scale(int64_t n3, const double *__restrict__ nd, double *v0)
{
    int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (k >= n3) return;
    const double den = nd[1];
    if (!(den > 0.0)) return;
    const double alpha = nd[0] / den;
    if (isfinite(alpha)) v0[k] *= alpha;
}

// Per-block partial of a weight gradient over the block's CHUNK nodes.  The
// first and the last layer, one side A of 64 columns and one side B of K: G =
// sum_n A[n][f] B[n][k] (AZ: A is dZ, f the output; else B is), and the bias
// gradient, the sum of dZ, behind it.  A thread keeps column f against all K,
// over every fourth node, straight from memory.
template <int K, bool AZ>
__global__ void __launch_bounds__(TB) k_mp_wgrad_thin(int64_t n, const float *__restrict__ A, const float *__restrict__ B,
                                                      float *__restrict__ partial)
{
    constexpr int NS = TB / H, NG = K * H + (AZ ? H : K);
    __shared__ float sh[NS][(K + 1) * H];
    const int f = threadIdx.x % H, s = threadIdx.x / H;
    const int64_t n0 = (int64_t)blockIdx.x * CHUNK, n1 = n < n0 + CHUNK ? n : n0 + CHUNK;
    float acc[K + 1];
#pragma unroll
    for (int k = 0; k <= K; ++k) acc[k] = 0.f;
#pragma unroll 4
    for (int64_t i = n0 + s; i < n1; i += NS) {
        const float a = A[i * H + f];
#pragma unroll
        for (int k = 0; k < K; ++k) acc[k] = fmaf(a, B[i * K + k], acc[k]);
        if (AZ) acc[K] += a;
        else if (f < K) acc[K] += B[i * K + f];
    }
#pragma unroll
    for (int k = 0; k <= K; ++k) sh[s][k * H + f] = acc[k];
    __syncthreads();
    float *o = partial + (int64_t)blockIdx.x * NG;
    for (int g = threadIdx.x; g < NG; g += TB) {
        // G index: AZ: f * K + k, bias f; else k * H + f, bias k
        const bool bias = g >= K * H;
        const int at = bias ? K * H + g - K * H : AZ ? (g % K) * H + g / K : g;
        float t = 0.f;
#pragma unroll
        for (int q = 0; q < NS; ++q) t += sh[q][at];
        o[g] = t;
    }
}

// The same for the layers (64 outputs, 128 inputs), FMA bound: a thread keeps
// 4 outputs x 8 inputs (64 threads also a bias), three 16-byte shared loads
// per 32 FMAs, and has the next 16 nodes' rows in flight in registers.  1e5
// cells: 236 -> 51 us.
__global__ void __launch_bounds__(TB, 3) k_mp_wgrad_layer(int64_t n, const float *__restrict__ dZ, const float *__restrict__ X1,
                                                          const float *__restrict__ X2, float *__restrict__ partial)
{
    constexpr int TILE = 16, NG = H * H2 + H, NZ = TILE * H / 4 / TB, NX = TILE * H2 / 4 / TB;
    __shared__ __align__(16) float zs[TILE][H];
    __shared__ __align__(16) float xs[TILE][H2];
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    const int64_t n0 = (int64_t)blockIdx.x * CHUNK, n1 = n < n0 + CHUNK ? n : n0 + CHUNK;
    float acc[4][8], bias = 0.f;
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 8; ++v) acc[u][v] = 0.f;
    float4 zq[NZ], xq[NX];
    auto fetch = [&](int64_t t0) {
#pragma unroll
        for (int q = 0; q < NZ; ++q) {
            const int c = threadIdx.x + q * TB;
            const int64_t i = t0 + c / (H / 4);
            zq[q] = i < n1 ? reinterpret_cast<const float4 *>(dZ + i * H)[c % (H / 4)] : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int q = 0; q < NX; ++q) {
            const int c = threadIdx.x + q * TB, k = c % (H2 / 4);
            const int64_t i = t0 + c / (H2 / 4);
            const float *x = k < H / 4 ? X1 : X2;
            xq[q] = i < n1 ? reinterpret_cast<const float4 *>(x + i * H)[k % (H / 4)] : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    };
    fetch(n0);
    for (int64_t t0 = n0; t0 < n1; t0 += TILE) {
        __syncthreads();
#pragma unroll
        for (int q = 0; q < NZ; ++q) reinterpret_cast<float4 *>(&zs[0][0])[threadIdx.x + q * TB] = zq[q];
#pragma unroll
        for (int q = 0; q < NX; ++q) reinterpret_cast<float4 *>(&xs[0][0])[threadIdx.x + q * TB] = xq[q];
        __syncthreads();
        if (t0 + TILE < n1) fetch(t0 + TILE);
        if (threadIdx.x < H)
            for (int s = 0; s < TILE; ++s) bias += zs[s][threadIdx.x];
#pragma unroll 4
        for (int s = 0; s < TILE; ++s) {
            const float4 z = *reinterpret_cast<const float4 *>(&zs[s][4 * ty]);
            const float4 a = *reinterpret_cast<const float4 *>(&xs[s][4 * tx]);
            const float4 b = *reinterpret_cast<const float4 *>(&xs[s][H + 4 * tx]);
            const float zv[4] = {z.x, z.y, z.z, z.w}, xv[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
            for (int u = 0; u < 4; ++u) {
#pragma unroll
                for (int v = 0; v < 8; ++v) acc[u][v] = fmaf(zv[u], xv[v], acc[u][v]);
            }
        }
    }
    float *o = partial + (int64_t)blockIdx.x * NG;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        float *r = o + (4 * ty + u) * H2 + 4 * tx;
        *reinterpret_cast<float4 *>(r) = make_float4(acc[u][0], acc[u][1], acc[u][2], acc[u][3]);
        *reinterpret_cast<float4 *>(r + H) = make_float4(acc[u][4], acc[u][5], acc[u][6], acc[u][7]);
    }
    if (threadIdx.x < H) o[H * H2 + threadIdx.x] = bias;
}

// grad[off + g] = sum over blocks of partial[b][g]: 8 runs of blocks per
// column, each in order, then the runs in order.
__global__ void __launch_bounds__(TB) k_mp_wsum(int nblocks, int NG, const float *__restrict__ partial, int off_w, int off_b,
                                                int nw, float *grad)
{
    constexpr int R = TB / 32;
    __shared__ float sh[R][32];
    const int g = blockIdx.x * 32 + (threadIdx.x & 31), r = threadIdx.x >> 5;
    const int per = (nblocks + R - 1) / R, b1 = min(nblocks, (r + 1) * per);
    float s = 0.f;
    if (g < NG) {
#pragma unroll 8
        for (int b = r * per; b < b1; ++b) s += partial[(int64_t)b * NG + g];
    }
    sh[r][threadIdx.x & 31] = s;
    __syncthreads();
    if (r || g >= NG) return;
#pragma unroll
    for (int k = 1; k < R; ++k) s += sh[k][threadIdx.x];
    if (g < nw) grad[off_w + g] = s;
    else grad[off_b + (g - nw)] = s;
}

// Adam on the FP32 master weights; refresh the BF16 copies.
__global__ void k_mp_adam(int np, float *p, const float *__restrict__ g, float *m, float *v, __nv_bfloat16 *pb,
                          float lr, float b1, float b2, float eps, float c1, float c2)
{
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= np) return;
    if (lr > 0.f) {
        const float gk = g[k];
        const float mk = b1 * m[k] + (1.f - b1) * gk;
        const float vk = b2 * v[k] + (1.f - b2) * gk * gk;
        m[k] = mk;
        v[k] = vk;
        p[k] -= lr * (mk / c1) / (sqrtf(vk / c2) + eps);
    }
    pb[k] = __float2bfloat16_rn(p[k]);
}

}  // namespace

struct sgp_mpnn {
    int64_t n = 0;
    int64_t steps = 0;
    DBuf p, pb, g, m, v;              // master, BF16, gradient, Adam moments
    DBuf basis, x, hs, aggs, c, v0w;  // activations of the last prediction
    DBuf dh, du, dc, part, red;
    DBuf tmp;                         // 3 x 3n float64: e, Gamma e, Gamma v*
    DBuf forest;                      // workspace of the forest solve
    const sgp_matrix *M = nullptr;
};

static sgp_status mpnn_ensure(sgp_ctx *ctx, sgp_mpnn *N, int64_t n)
{
    const size_t nn = (size_t)std::max<int64_t>(n, 1);
    SGP_TRY(buf_ensure(ctx, N->basis, sizeof(double) * 9 * nn));
    SGP_TRY(buf_ensure(ctx, N->x, sizeof(float) * DIN * nn));
    SGP_TRY(buf_ensure(ctx, N->hs, sizeof(float) * 4 * H * nn));
    SGP_TRY(buf_ensure(ctx, N->aggs, sizeof(float) * 3 * H * nn));
    SGP_TRY(buf_ensure(ctx, N->c, sizeof(float) * KB * nn));
    SGP_TRY(buf_ensure(ctx, N->v0w, sizeof(double) * 3 * nn));
    SGP_TRY(buf_ensure(ctx, N->dh, sizeof(float) * H * nn));
    SGP_TRY(buf_ensure(ctx, N->du, sizeof(float) * H2 * nn));
    SGP_TRY(buf_ensure(ctx, N->dc, sizeof(float) * KB * nn));
    const int64_t nblk = (n + CHUNK - 1) / CHUNK + 1;
    SGP_TRY(buf_ensure(ctx, N->part, sizeof(float) * (size_t)nblk * (H * H2 + H)));
    SGP_TRY(buf_ensure(ctx, N->red, sizeof(double) * 2 * 1024 + 256));
    SGP_TRY(buf_ensure(ctx, N->tmp, sizeof(double) * 12 * nn));
    N->n = n;
    return SGP_OK;
}

// A forest solve whose wait gave up left NaN in the basis: reported by the calls
// that wait for the stream.
static sgp_status forest_check(sgp_ctx *ctx)
{
    return gave_up(ctx) ? sgp_fail(ctx, SGP_ERR_TIMEOUT, "mpnn: a bounded device wait gave up in a forest solve") : SGP_OK;
}

static unsigned red_blocks(int64_t cnt)
{
    return (unsigned)std::max<int64_t>(1, std::min<int64_t>(1024, (cnt + TB - 1) / TB));
}

template <int D1, int D2, int DOUT, bool TRANS, bool RELU, int NU>
static sgp_status dense_tiles(sgp_ctx *ctx, int64_t n, const float *X1, const float *X2, const __nv_bfloat16 *W,
                              const __nv_bfloat16 *b, const int32_t *row_ptr, float *Y)
{
    constexpr int DI = D1 + D2;
    constexpr size_t smem = sizeof(float) * ((size_t)DI * DOUT + (size_t)16 * NU * (DI + 4));
    auto kern = k_mp_dense<D1, D2, DOUT, TRANS, RELU, NU>;
    SGP_CUDA(ctx, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    const int64_t want = (n + 16 * NU - 1) / (16 * NU);
    // two blocks per SM (registers)
    const unsigned G = (unsigned)std::max<int64_t>(1, std::min<int64_t>(want, 2 * ctx->num_sms));
    LAUNCH(ctx, kern, G, TB, smem, n, X1, X2, W, b, row_ptr, Y);
    return SGP_OK;
}
// 128 nodes per tile while that fills two blocks per SM, else 64
template <int D1, int D2, int DOUT, bool TRANS, bool RELU>
static sgp_status dense(sgp_ctx *ctx, int64_t n, const float *X1, const float *X2, const __nv_bfloat16 *W,
                        const __nv_bfloat16 *b, const int32_t *row_ptr, float *Y)
{
    return n >= 2 * (int64_t)ctx->num_sms * 128 ? dense_tiles<D1, D2, DOUT, TRANS, RELU, 8>(ctx, n, X1, X2, W, b, row_ptr, Y)
                              : dense_tiles<D1, D2, DOUT, TRANS, RELU, 4>(ctx, n, X1, X2, W, b, row_ptr, Y);
}

template <int D1, int D2, int DOUT>
static sgp_status wgrad(sgp_ctx *ctx, sgp_mpnn *N, int64_t n, const float *dZ, const float *X1, const float *X2,
                        int off_w, int off_b)
{
    constexpr int DI = D1 + D2;
    constexpr int NG = DOUT * DI + DOUT;
    const unsigned nb = (unsigned)((n + CHUNK - 1) / CHUNK);
    float *part = bp<float>(N->part);
    if constexpr (D1 == H && D2 == H && DOUT == H)
        LAUNCH(ctx, k_mp_wgrad_layer, nb, TB, 0, n, dZ, X1, X2, part);
    else if constexpr (DOUT == H)
        LAUNCH(ctx, (k_mp_wgrad_thin<DI, true>), nb, TB, 0, n, dZ, X1, part);
    else
        LAUNCH(ctx, (k_mp_wgrad_thin<DOUT, false>), nb, TB, 0, n, X1, dZ, part);
    LAUNCH(ctx, k_mp_wsum, grid_for(NG, 32), TB, 0, (int)nb, NG, (const float *)part, off_w, off_b, DOUT * DI,
           bp<float>(N->g));
    return SGP_OK;
}

extern "C" {

sgp_status sgp_mpnn_create(sgp_ctx *ctx, const float *params, int64_t count, sgp_mpnn **out)
{
    if (!ctx || !out || !params) return SGP_ERR_INVALID_ARG;
    if (count != NPARAM)
        return sgp_fail(ctx, SGP_ERR_INVALID_ARG, "mpnn_create: expected %d parameters, got %lld", NPARAM,
                        (long long)count);
    SGP_CUDA(ctx, cudaSetDevice(ctx->device));
    sgp_mpnn *N = new sgp_mpnn();
    *out = N;
    SGP_TRY(buf_ensure(ctx, N->p, sizeof(float) * NPARAM));
    SGP_TRY(buf_ensure(ctx, N->pb, sizeof(__nv_bfloat16) * NPARAM));
    SGP_TRY(buf_ensure(ctx, N->g, sizeof(float) * NPARAM));
    SGP_TRY(buf_ensure(ctx, N->m, sizeof(float) * NPARAM));
    SGP_TRY(buf_ensure(ctx, N->v, sizeof(float) * NPARAM));
    SGP_CUDA(ctx, cudaMemcpyAsync(N->p.p, params, sizeof(float) * NPARAM, cudaMemcpyHostToDevice, ctx->stream));
    SGP_CUDA(ctx, cudaMemsetAsync(N->g.p, 0, sizeof(float) * NPARAM, ctx->stream));
    SGP_CUDA(ctx, cudaMemsetAsync(N->m.p, 0, sizeof(float) * NPARAM, ctx->stream));
    SGP_CUDA(ctx, cudaMemsetAsync(N->v.p, 0, sizeof(float) * NPARAM, ctx->stream));
    LAUNCH(ctx, k_mp_adam, grid_for(NPARAM, TB), TB, 0, NPARAM, bp<float>(N->p), (const float *)bp<float>(N->g),
           bp<float>(N->m), bp<float>(N->v), bp<__nv_bfloat16>(N->pb), 0.f, 0.9f, 0.999f, 1e-8f, 1.f, 1.f);
    SGP_CUDA(ctx, cudaStreamSynchronize(ctx->stream));  // params lives in caller memory
    return SGP_OK;
}

void sgp_mpnn_destroy(sgp_mpnn *N)
{
    if (!N) return;
    cudaDeviceSynchronize();
    DBuf *bufs[] = {&N->p, &N->pb, &N->g, &N->m, &N->v, &N->basis, &N->x, &N->hs, &N->aggs,
                    &N->c, &N->v0w, &N->dh, &N->du, &N->dc, &N->part, &N->red, &N->tmp, &N->forest};
    for (DBuf *b : bufs)
        if (b->p) cudaFree(b->p);
    delete N;
}

sgp_status sgp_mpnn_params(sgp_ctx *ctx, const sgp_mpnn *N, float *params, float *grads)
{
    if (!ctx || !N) return SGP_ERR_INVALID_ARG;
    if (params) SGP_CUDA(ctx, cudaMemcpyAsync(params, N->p.p, sizeof(float) * NPARAM, cudaMemcpyDeviceToHost, ctx->stream));
    if (grads) SGP_CUDA(ctx, cudaMemcpyAsync(grads, N->g.p, sizeof(float) * NPARAM, cudaMemcpyDeviceToHost, ctx->stream));
    SGP_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    SGP_TRY(forest_check(ctx));
    return SGP_OK;
}

}  // extern "C"

// The forward pass in the matrix's internal cell order: F (and v_prev) are
// taken from the caller's order into N->tmp[9n, 12n) (and the third basis
// vector); the output stays in N->v0w, in internal order.
static sgp_status mpnn_forward_internal(sgp_ctx *ctx, sgp_mpnn *N, const sgp_matrix *M, const sgp_factor *Fh,
                                        const double *F, const double *v_prev)
{
    if (!ctx || !N || !M || !Fh || !F) return SGP_ERR_INVALID_ARG;
    if (Fh->n != M->n) return sgp_fail(ctx, SGP_ERR_INVALID_ARG, "mpnn_forward: factor and matrix differ in size");
    SGP_CUDA(ctx, cudaSetDevice(ctx->device));
    const int64_t n = M->n;
    SGP_TRY(mpnn_ensure(ctx, N, n));
    N->M = M;
    if (n == 0) return SGP_OK;
    double *b0 = bp<double>(N->basis), *b1 = b0 + 3 * n, *b2 = b1 + 3 * n;
    double *Fi = bp<double>(N->tmp) + 9 * n;
    const int32_t *orig_of = bp<const int32_t>(M->orig_of);
    cudaEvent_t ev;
    SGP_TRY(kt_begin(ctx, SGP_KT_WARM_BASIS, &ev));
    LAUNCH(ctx, k_to_internal<double>, grid_for(n, TB), TB, 0, n, orig_of, F, Fi);
    // basis: block-Jacobi solve, spanning-forest solve, previous velocity
    SGP_TRY(matrix_block_jacobi(ctx, const_cast<sgp_matrix *>(M)));
    LAUNCH(ctx, k_mp_jacobi, grid_for(n, TB), TB, 0, n, bp<const double>(M->jac), (const double *)Fi, b0);
    SGP_CUDA(ctx, cudaMemcpyAsync(b1, Fi, sizeof(double) * 3 * n, cudaMemcpyDeviceToDevice, ctx->stream));
    SGP_TRY(tree_apply_inplace<double>(ctx, Fh, b1, nullptr, &N->forest));
    if (v_prev) LAUNCH(ctx, k_to_internal<double>, grid_for(n, TB), TB, 0, n, orig_of, v_prev, b2);
    else SGP_CUDA(ctx, cudaMemsetAsync(b2, 0, sizeof(double) * 3 * n, ctx->stream));
    double *red = bp<double>(N->red);
    unsigned *counter = reinterpret_cast<unsigned *>(red + 2 * 1024 + 8);
    double *mean_b1 = red + 2 * 1024;
    SGP_CUDA(ctx, cudaMemsetAsync(counter, 0, sizeof(unsigned), ctx->stream));
    const unsigned G = (unsigned)std::min<int64_t>(1024, (n + TB - 1) / TB);
    LAUNCH(ctx, k_mp_norm_sum, G, TB, 0, n, (const double *)b1, red, counter, mean_b1);
    float *x = bp<float>(N->x);
    LAUNCH(ctx, k_mp_features, grid_for(n, TB), TB, 0, n, (const double *)b0, (const double *)b1,
           (const double *)b2, bp<const int32_t>(M->row_ptr), (const double *)mean_b1, x);
    SGP_TRY(kt_end(ctx, SGP_KT_WARM_BASIS, ev));
    SGP_TRY(kt_begin(ctx, SGP_KT_WARM_LAYERS, &ev));
    // forward
    const __nv_bfloat16 *pb = bp<const __nv_bfloat16>(N->pb);
    float *hs = bp<float>(N->hs), *aggs = bp<float>(N->aggs);
    const int32_t *row_ptr = bp<const int32_t>(M->row_ptr), *col = bp<const int32_t>(M->col);
    SGP_TRY((dense<DIN, 0, H, false, true>(ctx, n, x, nullptr, pb + OFF_WIN, pb + OFF_BIN, row_ptr, hs)));
    for (int l = 0; l < 3; ++l) {
        float *h = hs + (int64_t)l * H * n, *a = aggs + (int64_t)l * H * n, *hn = hs + (int64_t)(l + 1) * H * n;
        LAUNCH(ctx, k_mp_agg, grid_for(16 * n, TB), TB, 0, n, row_ptr, col, (const float *)h, a);
        const int off = OFF_L0 + l * LAYER;
        SGP_TRY((dense<H, H, H, false, true>(ctx, n, h, a, pb + off, pb + off + H * H2, row_ptr, hn)));
    }
    LAUNCH(ctx, k_mp_out, (unsigned)((n + ON - 1) / ON), TB, 0, n, (const float *)(hs + 3 * H * n), pb + OFF_WOUT, pb + OFF_BOUT,
           (const double *)b0, (const double *)b1, (const double *)b2, bp<float>(N->c), bp<double>(N->v0w));
    SGP_TRY(kt_end(ctx, SGP_KT_WARM_LAYERS, ev));
    return SGP_OK;
}

extern "C" {

sgp_status sgp_mpnn_forward(sgp_ctx *ctx, sgp_mpnn *N, const sgp_matrix *M, const sgp_factor *Fh,
                            const double *F, const double *v_prev, double *v0)
{
    if (!v0) return SGP_ERR_INVALID_ARG;
    SGP_TRY(mpnn_forward_internal(ctx, N, M, Fh, F, v_prev));
    const int64_t n = M->n;
    if (n > 0)
        LAUNCH(ctx, k_to_caller<double>, grid_for(n, TB), TB, 0, n, bp<const int32_t>(M->orig_of),
               bp<const double>(N->v0w), v0);
    return SGP_OK;
}

sgp_status sgp_mpnn_backward(sgp_ctx *ctx, sgp_mpnn *N, const double *v_target, int32_t loss_kind, double *loss)
{
    if (!ctx || !N || !N->M) return SGP_ERR_INVALID_ARG;
    if (loss_kind != SGP_MPNN_LOSS_L2 && loss_kind != SGP_MPNN_LOSS_ENERGY)
        return sgp_fail(ctx, SGP_ERR_INVALID_ARG, "mpnn_backward: unknown loss");
    if (N->n > 0 && !v_target) return SGP_ERR_INVALID_ARG;
    SGP_CUDA(ctx, cudaSetDevice(ctx->device));
    const int64_t n = N->n;
    if (n == 0) {
        SGP_CUDA(ctx, cudaMemsetAsync(N->g.p, 0, sizeof(float) * NPARAM, ctx->stream));
        if (loss) *loss = 0.0;
        return SGP_OK;
    }
    const sgp_matrix *M = N->M;
    const double *b0 = bp<const double>(N->basis), *b1 = b0 + 3 * n, *b2 = b1 + 3 * n;
    const double *v0 = bp<const double>(N->v0w);
    double *red = bp<double>(N->red);
    unsigned *counter = reinterpret_cast<unsigned *>(red + 2 * 1024 + 8);
    double *nd = red + 2 * 1024 + 2, *lossout = red + 2 * 1024 + 4;
    double *e = bp<double>(N->tmp), *Ge = e + 3 * n, *Gt = Ge + 3 * n, *vt = Gt + 3 * n;
    LAUNCH(ctx, k_to_internal<double>, grid_for(n, TB), TB, 0, n, bp<const int32_t>(M->orig_of), v_target, vt);
    v_target = vt;
    const unsigned G = red_blocks(3 * n);
    LAUNCH(ctx, k_mp_diff, grid_for(3 * n, TB), TB, 0, 3 * n, v0, v_target, e);
    const double *g = e;
    if (loss_kind == SGP_MPNN_LOSS_ENERGY) {
        SGP_TRY(spmv64(ctx, M, e, Ge));
        SGP_TRY(spmv64(ctx, M, v_target, Gt));
        LAUNCH(ctx, k_mp_dot2, G, TB, 0, 3 * n, (const double *)e, (const double *)Ge, v_target, (const double *)Gt,
               red, counter, nd);
        g = Ge;
    } else {
        LAUNCH(ctx, k_mp_dot2, G, TB, 0, 3 * n, (const double *)e, (const double *)e, v_target, v_target, red,
               counter, nd);
    }
    LAUNCH(ctx, k_mp_ratio, 1, 32, 0, (const double *)nd, lossout);
    float *dc = bp<float>(N->dc), *dh = bp<float>(N->dh), *du = bp<float>(N->du);
    const float *hs = bp<const float>(N->hs), *aggs = bp<const float>(N->aggs), *x = bp<const float>(N->x);
    const __nv_bfloat16 *pb = bp<const __nv_bfloat16>(N->pb);
    LAUNCH(ctx, k_mp_dc, grid_for(n, TB), TB, 0, n, g, b0, b1, b2, (const double *)nd, dc);
    // output layer
    SGP_TRY((wgrad<H, 0, KB>(ctx, N, n, dc, hs + 3 * H * n, nullptr, OFF_WOUT, OFF_BOUT)));
    const int32_t *row_ptr = bp<const int32_t>(M->row_ptr), *col = bp<const int32_t>(M->col);
    LAUNCH(ctx, k_mp_out_t, grid_for(16 * n, TB), TB, 0, n, (const float *)dc, pb + OFF_WOUT, hs + 3 * H * n, dh);
    for (int l = 2; l >= 0; --l) {
        const float *h = hs + (int64_t)l * H * n, *a = aggs + (int64_t)l * H * n;
        const int off = OFF_L0 + l * LAYER;
        SGP_TRY((wgrad<H, H, H>(ctx, N, n, dh, h, a, off, off + H * H2)));
        SGP_TRY((dense<H, 0, H2, true, false>(ctx, n, dh, nullptr, pb + off, nullptr, row_ptr, du)));
        LAUNCH(ctx, k_mp_agg_t, grid_for(16 * n, TB), TB, 0, n, row_ptr, col, (const float *)du, h, dh);
    }
    SGP_TRY((wgrad<DIN, 0, H>(ctx, N, n, dh, x, nullptr, OFF_WIN, OFF_BIN)));
    if (loss) {
        SGP_TRY(read_back(ctx, loss, lossout, sizeof(double)));
        SGP_TRY(forest_check(ctx));
    }
    return SGP_OK;
}

sgp_status sgp_mpnn_step(sgp_ctx *ctx, sgp_mpnn *N, float lr)
{
    if (!ctx || !N) return SGP_ERR_INVALID_ARG;
    if (!(lr > 0.f) || !std::isfinite(lr))
        return sgp_fail(ctx, SGP_ERR_INVALID_ARG, "mpnn_step: learning rate must be positive");
    SGP_CUDA(ctx, cudaSetDevice(ctx->device));
    N->steps++;
    const float c1 = 1.f - powf(0.9f, (float)N->steps);
    const float c2 = 1.f - powf(0.999f, (float)N->steps);
    LAUNCH(ctx, k_mp_adam, grid_for(NPARAM, TB), TB, 0, NPARAM, bp<float>(N->p), bp<const float>(N->g),
           bp<float>(N->m), bp<float>(N->v), bp<__nv_bfloat16>(N->pb), lr, 0.9f, 0.999f, 1e-8f, c1, c2);
    return SGP_OK;
}

}  // extern "C"

// The residual check of the warm start lives with the solver's product; it
// closes the timing bracket `ev` of class kclass before its read-back.
sgp_status mpnn_residual_check(sgp_ctx *ctx, const sgp_matrix *M, const double *F, double *v0, int *used,
                               int kclass, cudaEvent_t ev);

extern "C" sgp_status sgp_warm_start(sgp_ctx *ctx, sgp_mpnn *N, const sgp_matrix *M, const sgp_factor *Fh,
                                     const double *F, const double *v_prev, double *v0, int32_t flags,
                                     int32_t *used)
{
    if (flags & ~SGP_WARM_MR_SCALE) return sgp_fail(ctx, SGP_ERR_INVALID_ARG, "warm_start: unknown flags");
    if (!v0) return SGP_ERR_INVALID_ARG;
    SGP_TRY(mpnn_forward_internal(ctx, N, M, Fh, F, v_prev));
    const int64_t n = M->n;
    if (n == 0) {
        if (used) *used = 0;
        return SGP_OK;
    }
    // scaling and acceptance on a copy of the network output (internal order);
    // N->v0w stays the network's own output for a following backward pass
    double *Gv = bp<double>(N->tmp), *w = Gv + 3 * n;
    const double *Fi = bp<const double>(N->tmp) + 9 * n;
    cudaEvent_t ev;
    SGP_TRY(kt_begin(ctx, SGP_KT_WARM_CHECK, &ev));
    SGP_CUDA(ctx, cudaMemcpyAsync(w, N->v0w.p, sizeof(double) * 3 * n, cudaMemcpyDeviceToDevice, ctx->stream));
    int u = 0;
    bool checked = false;
    if (flags & SGP_WARM_MR_SCALE) {
        double *red = bp<double>(N->red);
        unsigned *counter = reinterpret_cast<unsigned *>(red + 2 * 1024 + 8);
        double *nd = red + 2 * 1024 + 2;
        SGP_TRY(spmv64(ctx, M, w, Gv));
        LAUNCH(ctx, k_mp_dot2, red_blocks(3 * n), TB, 0, 3 * n, (const double *)Gv, Fi, (const double *)Gv,
               (const double *)Gv, red, counter, nd);
        LAUNCH(ctx, k_mp_scale, grid_for(3 * n, TB), TB, 0, 3 * n, (const double *)nd, w);
        // with a finite step alpha = (Gamma v0)^T F / |Gamma v0|^2 the scaled
        // guess has |F - alpha Gamma v0|^2 = |F|^2 - ((Gamma v0)^T F)^2 /
        // |Gamma v0|^2 <= |F|^2: the acceptance test holds without a second
        // product
        SGP_TRY(kt_end(ctx, SGP_KT_WARM_CHECK, ev));
        double h[2] = {0.0, 0.0};
        SGP_TRY(read_back(ctx, h, nd, sizeof(h)));
        if (h[1] > 0.0 && std::isfinite(h[0] / h[1])) {
            u = 1;
            checked = true;
        } else {
            SGP_TRY(kt_begin(ctx, SGP_KT_WARM_CHECK, &ev));
        }
    }
    if (!checked) SGP_TRY(mpnn_residual_check(ctx, M, Fi, w, &u, SGP_KT_WARM_CHECK, ev));
    LAUNCH(ctx, k_to_caller<double>, grid_for(n, TB), TB, 0, n, bp<const int32_t>(M->orig_of), (const double *)w,
           v0);
    if (used) *used = u;
    return forest_check(ctx);   // (a read-back lies behind the forest solve)
}
