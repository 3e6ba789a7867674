// Learned initial density for the SCF (the paper starts from a superposition of atomic densities,
// Sec. 2.1, and lists machine learning as future work, Sec. 4): a 32 -> 64 -> 64 -> 1 SiLU network
// on atom-centred radial descriptors predicts rho* - rho_SAD at every grid point.
//
//   G_j(x) = sum_a sum_T exp(-(r - mu_j)^2 / (2 eta^2)) f_c(r), r = |x - R_a - T| <= 6.5 bohr,
//   f_c(r) = (cos(pi r / 6.5) + 1)/2, mu_j = 6 j/31, eta = 6/31.
//
// Features are stored in BF16; the forward and backward passes use BF16-rounded weights with
// FP32 activations and accumulation; Adam keeps FP32 master weights and moments.
// Training kernel: persistent CTAs, 128-point tiles; activations of a tile live in shared memory, the CTA's
// weight gradients in registers, and they are added to the global gradient once.
#include "internal.cuh"

#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstddef>

namespace sdft {
namespace {

constexpr int NF = 32, NH = 64;
constexpr int OW1 = 0, OB1 = OW1 + NH * NF, OW2 = OB1 + NH, OB2 = OW2 + NH * NH, OW3 = OB2 + NH, OB3 = OW3 + NH;
constexpr int NP = OB3 + 1;   // 6337 parameters
constexpr int TP = 128;       // points per tile

// silu(z) = z s, s = 1 / (1 + e^-z), and (TRAIN) silu'(z) = s (1 + z (1 - s)) in place of z: one exponential and one
// division for both
template <bool TRAIN>
__device__ __forceinline__ float activate(float& z) {
    const float s = 1.f / (1.f + __expf(-z)), h = z * s;
    if (TRAIN) z = s * (1.f + z * (1.f - s));
    return h;
}
template <bool TRAIN>
__device__ __forceinline__ float2 activate(float2& z) {
    const float x = activate<TRAIN>(z.x), y = activate<TRAIN>(z.y);
    return make_float2(x, y);
}
// packed FP32 pair multiply-add (Blackwell f32x2): a .* b + c
__device__ __forceinline__ float2 ffma2(float2 a, float2 b, float2 c) {
    unsigned long long r, ua, ub, uc;
    asm("mov.b64 %0, {%1, %2};" : "=l"(ua) : "f"(a.x), "f"(a.y));
    asm("mov.b64 %0, {%1, %2};" : "=l"(ub) : "f"(b.x), "f"(b.y));
    asm("mov.b64 %0, {%1, %2};" : "=l"(uc) : "f"(c.x), "f"(c.y));
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(ua), "l"(ub), "l"(uc));
    float2 o;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(o.x), "=f"(o.y) : "l"(r));
    return o;
}
__device__ __forceinline__ float bf16r(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

// ---- network kernels -------------------------------------------------------------------
// One CTA takes tiles of 128 points through the whole network, and back for training.  Every layer and every
// weight gradient is an FP32 product with both operands in shared memory, laid out so that each thread reads
// 16-byte vectors along both of its output dimensions: a forward thread owns 8 points x 4 neurons (3 vector loads
// for 32 multiply-adds, issued as packed pairs of points, fma.rn.f32x2), a gradient thread 8 x 8 weights of W2 and
// 8 x 4 of W1 over a quarter of the tile's points (4 + 3 loads for 64 + 32).  The forward sums add their terms in
// the same order as a plain loop over the inputs.  Activations are written twice where a product needs them along
// points (next layer) and along neurons (gradient).  Weight gradients stay in registers over all tiles of the CTA.
// The kernel this replaces read two scalars from shared memory for every multiply-add of a gradient and kept the
// gradient there too: 65 536 points, loss and gradient: 255 -> 81 us;
// 512 000 points, inference: 443 -> 190 us.
constexpr int MT = 256;              // threads
constexpr int XS = NF + 4, HS = NH + 4;   // row strides of the point-major copies (conflict-free vector stores)
struct MlpSmem {
    float W1T[NF][NH];   // W1 transposed (bf16-rounded)
    float W2T[NH][NH];   // W2T[g][h] = W2[h][g]
    float W2N[NH][NH];   // W2 itself (backward)
    float b1[NH], b2[NH], w3[NH];
    float b3;
    int pad[3];
    float Xt[NF][TP];    // features, along points
    float A[NH][TP];     // H1, then dZ2, along points
    float X[TP][XS];     // features, along inputs        (training only from here on)
    float H1[TP][HS];
    float dZ2[TP][HS];
    float dZ1[TP][HS];
};
constexpr size_t MLP_SMEM_FWD = offsetof(MlpSmem, X);

// acc[point pair][neuron] += x[8 points] w[4 neurons]
__device__ __forceinline__ void fma_8x4(float2 (&acc)[4][4], const float4 xa, const float4 xb, const float4 w) {
    const float2 x[4] = {make_float2(xa.x, xa.y), make_float2(xa.z, xa.w), make_float2(xb.x, xb.y), make_float2(xb.z, xb.w)};
    const float wv[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
    for (int n = 0; n < 4; ++n) {
        const float2 ww = make_float2(wv[n], wv[n]);
#pragma unroll
        for (int p = 0; p < 4; ++p) acc[p][n] = ffma2(x[p], ww, acc[p][n]);
    }
}
// acc over K rows of a point-major-along-columns operand `at` [K][TP] and weights `wt` [K][NH]
template <int K>
__device__ __forceinline__ void product_8x4(float2 (&acc)[4][4], const float (*at)[TP], const float (*wt)[NH], int p0, int n0) {
#pragma unroll 4
    for (int k = 0; k < K; ++k)
        fma_8x4(acc, *reinterpret_cast<const float4*>(&at[k][p0]), *reinterpret_cast<const float4*>(&at[k][64 + p0]),
                *reinterpret_cast<const float4*>(&wt[k][n0]));
}
// points of value pair p, half h: p0 + {0..3} and 64 + p0 + {0..3}
__device__ __forceinline__ int pt8(int p0, int i) { return (i < 4 ? 0 : 60) + p0 + i; }
__device__ __forceinline__ float& el(float2 (&a)[4][4], int i, int n) { return (i & 1) ? a[i >> 1][n].y : a[i >> 1][n].x; }

// store 8 x 4 values along points (rows of neurons) and, P != null, along neurons (rows of points)
__device__ __forceinline__ void store_8x4(float2 (&v)[4][4], float (*at)[TP], float (*pm)[HS], int p0, int n0) {
    if (at) {
#pragma unroll
        for (int n = 0; n < 4; ++n) {
            *reinterpret_cast<float4*>(&at[n0 + n][p0]) = make_float4(v[0][n].x, v[0][n].y, v[1][n].x, v[1][n].y);
            *reinterpret_cast<float4*>(&at[n0 + n][64 + p0]) = make_float4(v[2][n].x, v[2][n].y, v[3][n].x, v[3][n].y);
        }
    }
    if (pm) {
#pragma unroll
        for (int i = 0; i < 8; ++i)
            *reinterpret_cast<float4*>(&pm[pt8(p0, i)][n0]) = make_float4(el(v, i, 0), el(v, i, 1), el(v, i, 2), el(v, i, 3));
    }
}

// TRAIN: accumulate d(mean loss)/d(params) into grad (global, FP32) and the loss sum into loss.
// !TRAIN: y = network output.
// TRAIN visits the batch points perm((start + i) mod npts), i < nb, perm(j) = j * mult mod npts
// (mult coprime to npts); inference visits points 0 .. nb-1 in order.
template <bool TRAIN>
__global__ void __launch_bounds__(MT, TRAIN ? 1 : 2)
mlp_tile_kernel(const __nv_bfloat16* __restrict__ feat, const float* __restrict__ target, long long npts, long long nb,
                long long start, long long mult, const float* __restrict__ params, float* __restrict__ y_out,
                float* __restrict__ grad, double* __restrict__ loss, double inv_n) {
    extern __shared__ __align__(16) unsigned char smraw[];
    MlpSmem& S = *reinterpret_cast<MlpSmem*>(smraw);
    __shared__ long long pidx[TP];
    __shared__ float ypart[4][TP], dys[TP];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int q = tid; q < NH * NF; q += MT) S.W1T[q % NF][q / NF] = bf16r(params[OW1 + q]);
    for (int q = tid; q < NH * NH; q += MT) {
        const int h = q / NH, g = q - h * NH;
        const float w = bf16r(params[OW2 + q]);
        S.W2T[g][h] = w;
        if (TRAIN) S.W2N[h][g] = w;
    }
    for (int q = tid; q < NH; q += MT) {
        S.b1[q] = bf16r(params[OB1 + q]);
        S.b2[q] = bf16r(params[OB2 + q]);
        S.w3[q] = bf16r(params[OW3 + q]);
    }
    if (tid == 0) S.b3 = bf16r(params[OB3]);
    __syncthreads();
    // forward tile of the thread: points p0.., 64 + p0.., neurons n0..n0+3
    const int quad = warp >> 1;                                  // 16 neurons
    const int n0 = quad * 16 + (lane & 3) * 4;
    const int p0 = ((warp & 1) * 8 + (lane >> 2)) * 4;
    // gradient tile of the thread: points of quarter kq, W2 rows 4 hi.., 32 + 4 hi.., columns 4 gi.., 32 + 4 gi..;
    // W1 the same rows, columns 4 gi..
    const int kq = tid >> 6, hi = (tid >> 3) & 7, gi = tid & 7;
    float2 gw2[8][4];   // [row][column pair]
    float2 gw1[8][2];
    float gb1[4] = {0, 0, 0, 0}, gb2[4] = {0, 0, 0, 0}, gw3[4] = {0, 0, 0, 0}, gb3 = 0.f;
    if (TRAIN) {
#pragma unroll
        for (int a = 0; a < 8; ++a) {
#pragma unroll
            for (int b = 0; b < 4; ++b) gw2[a][b] = make_float2(0.f, 0.f);
#pragma unroll
            for (int b = 0; b < 2; ++b) gw1[a][b] = make_float2(0.f, 0.f);
        }
    }
    double lsum = 0.0;
    const bool vec = (reinterpret_cast<uintptr_t>(feat) & 15) == 0;   // 16-byte loads of a point's features
    const long long ntile = (nb + TP - 1) / TP;
    for (long long tile = blockIdx.x; tile < ntile; tile += gridDim.x) {
        const long long t0 = tile * TP;
        const int np = (int)(nb - t0 < TP ? nb - t0 : TP);
        if (tid < TP) {
            long long g = t0 + tid;
            if (TRAIN && tid < np) g = (((start + g) % npts) * mult) % npts;
            pidx[tid] = g;
        }
        __syncthreads();
        {   // features: two threads per point, 16 inputs each
            const int p = tid & (TP - 1), f0 = (tid / TP) * 16;
            float v[16];
            if (p < np && !vec) {
#pragma unroll
                for (int k = 0; k < 16; ++k) v[k] = __bfloat162float(feat[pidx[p] * NF + f0 + k]);
            } else if (p < np) {
                const uint4* src = reinterpret_cast<const uint4*>(feat + pidx[p] * NF + f0);
                const uint4 u[2] = {src[0], src[1]};
                const unsigned* w = reinterpret_cast<const unsigned*>(u);
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    v[2 * k] = __uint_as_float(w[k] << 16);
                    v[2 * k + 1] = __uint_as_float(w[k] & 0xffff0000u);
                }
            } else {
#pragma unroll
                for (int k = 0; k < 16; ++k) v[k] = 0.f;
            }
#pragma unroll
            for (int k = 0; k < 16; ++k) S.Xt[f0 + k][p] = v[k];
            if (TRAIN) {
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    *reinterpret_cast<float4*>(&S.X[p][f0 + 4 * k]) = make_float4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
            }
        }
        __syncthreads();
        float2 z1[4][4], z2[4][4];
        // layer 1: Z1 = X W1^T + b1
#pragma unroll
        for (int n = 0; n < 4; ++n)
#pragma unroll
            for (int p = 0; p < 4; ++p) z1[p][n] = make_float2(S.b1[n0 + n], S.b1[n0 + n]);
        product_8x4<NF>(z1, S.Xt, S.W1T, p0, n0);
        {
            float2 h[4][4];
#pragma unroll
            for (int p = 0; p < 4; ++p)
#pragma unroll
                for (int n = 0; n < 4; ++n) h[p][n] = activate<TRAIN>(z1[p][n]);   // z1 <- silu'(z1)
            store_8x4(h, S.A, TRAIN ? S.H1 : nullptr, p0, n0);
        }
        __syncthreads();
        // layer 2: Z2 = H1 W2^T + b2
#pragma unroll
        for (int n = 0; n < 4; ++n)
#pragma unroll
            for (int p = 0; p < 4; ++p) z2[p][n] = make_float2(S.b2[n0 + n], S.b2[n0 + n]);
        product_8x4<NH>(z2, S.A, S.W2T, p0, n0);
        // output: y = silu(Z2) . w3 + b3
        float2 h2[4][4];
        float w3[4];
#pragma unroll
        for (int n = 0; n < 4; ++n) w3[n] = S.w3[n0 + n];
#pragma unroll
        for (int p = 0; p < 4; ++p)
#pragma unroll
            for (int n = 0; n < 4; ++n) h2[p][n] = activate<TRAIN>(z2[p][n]);          // z2 <- silu'(z2)
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            float s = 0.f;
#pragma unroll
            for (int n = 0; n < 4; ++n) s = fmaf(el(h2, i, n), w3[n], s);
            s += __shfl_xor_sync(0xffffffffu, s, 1);
            s += __shfl_xor_sync(0xffffffffu, s, 2);
            if ((lane & 3) == 0) ypart[quad][pt8(p0, i)] = s;
        }
        __syncthreads();
        if (tid < TP) {
            const float y = ((ypart[0][tid] + ypart[1][tid]) + (ypart[2][tid] + ypart[3][tid])) + S.b3;
            if (!TRAIN) {
                if (tid < np) y_out[t0 + tid] = y;
            } else {
                const float e = tid < np ? y - target[pidx[tid]] : 0.f;
                lsum += (double)e * e;
                const float d = (float)(2.0 * inv_n) * e;
                dys[tid] = d;
                gb3 += d;
            }
        }
        __syncthreads();
        if (TRAIN) {
            // dZ2 = dy w3 silu'(Z2), with d w3, d b2
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const float dy = dys[pt8(p0, i)];
#pragma unroll
                for (int n = 0; n < 4; ++n) {
                    gw3[n] = fmaf(dy, el(h2, i, n), gw3[n]);
                    const float d = dy * w3[n] * el(z2, i, n);
                    gb2[n] += d;
                    el(h2, i, n) = d;
                }
            }
            store_8x4(h2, S.A, S.dZ2, p0, n0);   // every read of H1 along points is behind a barrier
            __syncthreads();
            // dZ1 = (dZ2 W2) silu'(Z1), with d b1
            {
                float2 a[4][4];
#pragma unroll
                for (int p = 0; p < 4; ++p)
#pragma unroll
                    for (int n = 0; n < 4; ++n) a[p][n] = make_float2(0.f, 0.f);
                product_8x4<NH>(a, S.A, S.W2N, p0, n0);
#pragma unroll
                for (int p = 0; p < 4; ++p)
#pragma unroll
                    for (int n = 0; n < 4; ++n) {
                        a[p][n].x *= z1[p][n].x;
                        a[p][n].y *= z1[p][n].y;
                        gb1[n] += a[p][n].x + a[p][n].y;
                    }
                store_8x4(a, nullptr, S.dZ1, p0, n0);
            }
            // d W2[h][g] = sum_p dZ2[p][h] H1[p][g] over this quarter of the points
#pragma unroll 2
            for (int p = kq * (TP / 4); p < (kq + 1) * (TP / 4); ++p) {
                const float4 da = *reinterpret_cast<const float4*>(&S.dZ2[p][4 * hi]);
                const float4 db = *reinterpret_cast<const float4*>(&S.dZ2[p][32 + 4 * hi]);
                const float4 ha = *reinterpret_cast<const float4*>(&S.H1[p][4 * gi]);
                const float4 hb = *reinterpret_cast<const float4*>(&S.H1[p][32 + 4 * gi]);
                const float d[8] = {da.x, da.y, da.z, da.w, db.x, db.y, db.z, db.w};
                const float2 h[4] = {make_float2(ha.x, ha.y), make_float2(ha.z, ha.w), make_float2(hb.x, hb.y), make_float2(hb.z, hb.w)};
#pragma unroll
                for (int r = 0; r < 8; ++r)
#pragma unroll
                    for (int q = 0; q < 4; ++q) gw2[r][q] = ffma2(make_float2(d[r], d[r]), h[q], gw2[r][q]);
            }
            __syncthreads();
            // d W1[h][f] = sum_p dZ1[p][h] X[p][f]
#pragma unroll 2
            for (int p = kq * (TP / 4); p < (kq + 1) * (TP / 4); ++p) {
                const float4 da = *reinterpret_cast<const float4*>(&S.dZ1[p][4 * hi]);
                const float4 db = *reinterpret_cast<const float4*>(&S.dZ1[p][32 + 4 * hi]);
                const float4 x = *reinterpret_cast<const float4*>(&S.X[p][4 * gi]);
                const float d[8] = {da.x, da.y, da.z, da.w, db.x, db.y, db.z, db.w};
#pragma unroll
                for (int r = 0; r < 8; ++r) {
                    gw1[r][0] = ffma2(make_float2(d[r], d[r]), make_float2(x.x, x.y), gw1[r][0]);
                    gw1[r][1] = ffma2(make_float2(d[r], d[r]), make_float2(x.z, x.w), gw1[r][1]);
                }
            }
            __syncthreads();   // X and the activations are free for the next tile
        }
    }
    if (TRAIN) {
        // sum the CTA's gradient in shared memory (over the activations, free now): the four point quarters one after
        // another, then the per-neuron sums of the 16 point groups; one addition to the global gradient per parameter
        float* acc = &S.Xt[0][0];
        static_assert(sizeof(float) * NP <= sizeof(S.Xt) + sizeof(S.A), "gradient scratch");
        for (int q = tid; q < NP; q += MT) acc[q] = 0.f;
        __syncthreads();
        for (int k = 0; k < 4; ++k) {
            if (kq == k) {
#pragma unroll
                for (int r = 0; r < 8; ++r) {
                    const int h = (r < 4 ? 0 : 28) + 4 * hi + r;
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const int g = (q < 2 ? 0 : 28) + 4 * gi + 2 * q;
                        acc[OW2 + h * NH + g] += gw2[r][q].x;
                        acc[OW2 + h * NH + g + 1] += gw2[r][q].y;
                    }
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        acc[OW1 + h * NF + 4 * gi + 2 * q] += gw1[r][q].x;
                        acc[OW1 + h * NF + 4 * gi + 2 * q + 1] += gw1[r][q].y;
                    }
                }
            }
            __syncthreads();
        }
#pragma unroll
        for (int n = 0; n < 4; ++n) {
            for (int off = 16; off >= 4; off >>= 1) {   // the warp's 8 point groups of a neuron
                gb1[n] += __shfl_down_sync(0xffffffffu, gb1[n], off);
                gb2[n] += __shfl_down_sync(0xffffffffu, gb2[n], off);
                gw3[n] += __shfl_down_sync(0xffffffffu, gw3[n], off);
            }
        }
        for (int half = 0; half < 2; ++half) {
            if ((warp & 1) == half && lane < 4) {
#pragma unroll
                for (int n = 0; n < 4; ++n) {
                    acc[OB1 + n0 + n] += gb1[n];
                    acc[OB2 + n0 + n] += gb2[n];
                    acc[OW3 + n0 + n] += gw3[n];
                }
            }
            __syncthreads();
        }
        if (tid < TP) {
            for (int off = 16; off > 0; off >>= 1) gb3 += __shfl_down_sync(0xffffffffu, gb3, off);
            if (lane == 0) ypart[0][warp] = gb3;
        }
        __syncthreads();
        if (tid == 0) acc[OB3] = (ypart[0][0] + ypart[0][1]) + (ypart[0][2] + ypart[0][3]);
        __syncthreads();
        for (int q = tid; q < NP; q += MT) atomicAdd(&grad[q], acc[q]);
        for (int off = 16; off > 0; off >>= 1) lsum += __shfl_down_sync(0xffffffffu, lsum, off);
        if (lane == 0 && tid < TP) atomicAdd(loss, lsum * inv_n);
    }
}

__global__ void adam_kernel(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                            float* __restrict__ v, int n, float lr, float b1, float b2, float eps, float c1, float c2) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const float gi = g[i];
        const float mi = b1 * m[i] + (1.f - b1) * gi;
        const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    }
}

__global__ void guess_kernel(const double* __restrict__ sad, const float* __restrict__ y, double* __restrict__ out,
                             long long n) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        out[i] = fmax(sad[i] + (double)y[i], 0.0);
}

__global__ void scale_kernel(double* __restrict__ x, const double* __restrict__ s, double nelec_over_dv, long long n) {
    const double f = nelec_over_dv / s[0];
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        x[i] *= f;
}

__global__ void sum_kernel(const double* __restrict__ x, long long n, double* __restrict__ out) {
    __shared__ double sh[32];
    double s = 0.0;
    for (long long i = threadIdx.x; i < n; i += blockDim.x) s += x[i];
    for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += sh[w];
        out[0] = t;
    }
}

__global__ void split_kernel(const double* __restrict__ rho, int nspin, double moment, double* __restrict__ out,
                             long long n) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        if (nspin == 1) {
            out[i] = rho[i];
        } else {
            out[i] = 0.5 * rho[i] * (1.0 + moment);
            out[n + i] = 0.5 * rho[i] * (1.0 - moment);
        }
    }
}

__global__ void target_kernel(const double* __restrict__ rho, int nspin, const double* __restrict__ sad,
                              float* __restrict__ t, long long n) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        double r = rho[i];
        if (nspin == 2) r += rho[n + i];
        t[i] = (float)(r - sad[i]);
    }
}

size_t tile_smem(bool train) { return train ? sizeof(MlpSmem) : MLP_SMEM_FWD; }

int tile_grid(cudaStream_t) {
    int dev = 0, nsm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    return std::max(1, nsm);
}

}  // namespace

int mlp_nparam() { return NP; }

// features of every grid point of the context's cell; target (optional) = rho_out - rho_SAD of the
// last SCF, summed over spins
void mlp_dataset(sdft_ctx* c, void* feat, float* target) {
    descriptor_field(c, feat);
    if (target) {
        target_kernel<<<(unsigned)std::min<long long>((c->ng + 255) / 256, 152LL * 16), 256, 0, c->stream>>>(
            c->rho_out, c->opt.nspin, c->rho_sad, target, c->ng);
        SDFT_CUDA(cudaGetLastError());
        count_launch(c);
    }
    SDFT_CUDA(cudaStreamSynchronize(c->stream));
}

long long perm_mult(long long npts) { return npts % 1000003LL == 0 ? 999983LL : 1000003LL; }

// grad (FP32 [NP]) is overwritten; the batch's mean squared error is added to *loss (device)
void mlp_loss_grad(const void* feat, const float* target, long long npts, long long batch, long long start,
                   const float* params, float* grad, double* loss, cudaStream_t st) {
    SDFT_CUDA(cudaMemsetAsync(grad, 0, sizeof(float) * NP, st));
    const size_t sm = tile_smem(true);
    allow_dynamic_smem(mlp_tile_kernel<true>, sm);
    const long long ntile = (batch + TP - 1) / TP;
    const int grid = (int)std::min<long long>(ntile, tile_grid(st));
    mlp_tile_kernel<true><<<grid, MT, sm, st>>>(reinterpret_cast<const __nv_bfloat16*>(feat), target, npts, batch,
                                                  start % npts, perm_mult(npts), params, nullptr, grad, loss,
                                                  1.0 / (double)batch);
    SDFT_CUDA(cudaGetLastError());
}

void mlp_forward(const void* feat, long long npts, const float* params, float* y, cudaStream_t st) {
    const size_t sm = tile_smem(false);
    allow_dynamic_smem(mlp_tile_kernel<false>, sm);
    const long long ntile = (npts + TP - 1) / TP;
    const int grid = (int)std::min<long long>(ntile, 2LL * tile_grid(st));
    mlp_tile_kernel<false><<<grid, MT, sm, st>>>(reinterpret_cast<const __nv_bfloat16*>(feat), nullptr, npts, npts,
                                                   0, 1, params, y, nullptr, nullptr, 1.0);
    SDFT_CUDA(cudaGetLastError());
}

void mlp_adam(float* p, const float* g, float* m, float* v, int step, double lr, cudaStream_t st) {
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.f - powf(b1, (float)step), c2 = 1.f - powf(b2, (float)step);
    adam_kernel<<<(NP + 255) / 256, 256, 0, st>>>(p, g, m, v, NP, (float)lr, b1, b2, 1e-8f, c1, c2);
    SDFT_CUDA(cudaGetLastError());
}

// nsteps of mini-batch Adam; step s (counted from first_step) uses the batch starting at
// (s - 1) * batch; loss_dev[s - first_step] receives that batch's loss before the update
void mlp_train(const void* feat, const float* target, long long npts, long long batch, float* params, float* grad,
               float* m, float* v, int first_step, int nsteps, double lr, double* loss_dev, cudaStream_t st) {
    SDFT_CUDA(cudaMemsetAsync(loss_dev, 0, sizeof(double) * nsteps, st));
    for (int k = 0; k < nsteps; ++k) {
        const int step = first_step + k;
        const long long start = (long long)((((unsigned long long)(step - 1)) * (unsigned long long)batch) %
                                            (unsigned long long)npts);
        mlp_loss_grad(feat, target, npts, batch, start, params, grad, loss_dev + k, st);
        mlp_adam(params, grad, m, v, step, lr, st);
    }
}

// rho_guess = max(rho_SAD + y, 0) renormalised to N_e, split into spins, stored as the user guess
void mlp_guess(sdft_ctx* c, const float* params) {
    const long long ng = c->ng;
    if (!c->mlp_scratch) c->mlp_scratch = ctx_alloc(c, (size_t)ng * (NF * 2 + sizeof(float)));
    void* feat = c->mlp_scratch;                                              // [ng][32] bf16
    float* y = reinterpret_cast<float*>(static_cast<char*>(c->mlp_scratch) + (size_t)ng * NF * 2);
    mlp_dataset(c, feat, nullptr);
    mlp_forward(feat, ng, params, y, c->stream);
    double* g = c->work64 + 8 * ng;
    guess_kernel<<<(unsigned)std::min<long long>((ng + 255) / 256, 152LL * 16), 256, 0, c->stream>>>(c->rho_sad, y, g,
                                                                                                    ng);
    sum_kernel<<<1, 1024, 0, c->stream>>>(g, ng, c->scal + 32);
    scale_kernel<<<(unsigned)std::min<long long>((ng + 255) / 256, 152LL * 16), 256, 0, c->stream>>>(
        g, c->scal + 32, c->nelec / c->dV, ng);
    SDFT_CUDA(cudaGetLastError());
    count_launch(c, 4);
    // spin split as for the SAD guess; the guess becomes the user density of the next SCF
    split_kernel<<<(unsigned)std::min<long long>((ng + 255) / 256, 152LL * 16), 256, 0, c->stream>>>(
        g, c->opt.nspin, c->opt.initial_moment, c->rho_user, ng);
    SDFT_CUDA(cudaGetLastError());
    count_launch(c);
    SDFT_CUDA(cudaMemcpyAsync(c->rho_in, c->rho_user, sizeof(double) * c->opt.nspin * ng, cudaMemcpyDeviceToDevice,
                              c->stream));
    c->user_density = true;
    SDFT_CUDA(cudaStreamSynchronize(c->stream));
}

}  // namespace sdft
