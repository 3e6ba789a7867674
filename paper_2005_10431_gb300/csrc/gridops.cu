// Grid-level FP64 kernels of the SCF (paper Sec. 2.1): Perdew-Zunger LDA, the AAR Poisson solver, density from
// orbitals (Eq. 2), Fermi-Dirac occupations, Pulay mixing, reductions and Hellmann-Feynman forces.
#include "internal.cuh"

#include <algorithm>
#include <cmath>
#include <cstring>

namespace sdft {
namespace {

constexpr int RB = 256;   // reduction block size

// an atom's pseudocharge amplitude, width and cut-off
struct AtomG {
    double pos[3];
    double amp_b, w_b, cut_b;
};

// ---------------------------------------------------------------------------------------
// reductions: deterministic two-stage sums of several dot products
// ---------------------------------------------------------------------------------------
struct DotArgs {
    const double* a[8];
    const double* b[8];
};
// K dots at once; the pointers come with the launch (no table upload), the K accumulators in registers
template <int K>
__global__ void __launch_bounds__(RB) multidot_kernel(const __grid_constant__ DotArgs P, long long n,
                                                      double* __restrict__ part) {
    double acc[K];
#pragma unroll
    for (int k = 0; k < K; ++k) acc[k] = 0.0;
    const long long step = (long long)gridDim.x * blockDim.x;
    long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    for (; i + 3 * step < n; i += 4 * step) {   // four points' loads in flight, added in order
        double x[4][K], y[4][K];
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int k = 0; k < K; ++k) {
                x[u][k] = P.a[k][i + u * step];
                y[u][k] = P.b[k][i + u * step];
            }
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int k = 0; k < K; ++k) acc[k] = fma(x[u][k], y[u][k], acc[k]);
    }
    for (; i < n; i += step) {
#pragma unroll
        for (int k = 0; k < K; ++k) acc[k] = fma(P.a[k][i], P.b[k][i], acc[k]);
    }
    __shared__ double sh[K][RB / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        double v = acc[k];
        for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
        if (lane == 0) sh[k][warp] = v;
    }
    __syncthreads();
    if (threadIdx.x < K) {
        double v = 0.0;
        for (int w = 0; w < RB / 32; ++w) v += sh[threadIdx.x][w];
        part[(long long)blockIdx.x * K + threadIdx.x] = v;
    }
}

// v + x[0] + x[stride] + ... (count terms, added one after another with `U` loads in flight)
template <int U>
__device__ __forceinline__ double ordered_sum(const double* __restrict__ x, int count, long long stride, double v = 0.0) {
    int s = 0;
    for (; s + U <= count; s += U) {
        double t[U];
#pragma unroll
        for (int u = 0; u < U; ++u) t[u] = x[(s + u) * stride];
#pragma unroll
        for (int u = 0; u < U; ++u) v += t[u];
    }
    for (; s < count; ++s) v += x[s * stride];
    return v;
}

__global__ void multidot_finish_kernel(const double* __restrict__ part, int nblk, int K, double* __restrict__ out) {
    const int k = threadIdx.x;
    if (k < K) out[k] = ordered_sum<32>(part + k, nblk, K);
}

// ---------------------------------------------------------------------------------------
// LDA (Perdew & Zunger 1981): PZ81 correlation, Dirac exchange, von Barth-Hedin f(zeta)
// ---------------------------------------------------------------------------------------
struct PZ {
    double g, b1, b2, A, B, C, D;
};
__device__ __forceinline__ void pz_phase(double rs, const PZ& p, double& eps, double& mu) {
    if (rs >= 1.0) {
        const double s = sqrt(rs);
        const double den = 1.0 + p.b1 * s + p.b2 * rs;
        eps = p.g / den;
        mu = eps * (1.0 + 7.0 / 6.0 * p.b1 * s + 4.0 / 3.0 * p.b2 * rs) / den;
    } else {
        const double lr = log(rs);
        eps = p.A * lr + p.B + p.C * rs * lr + p.D * rs;
        mu = p.A * lr + (p.B - p.A / 3.0) + 2.0 / 3.0 * p.C * rs * lr + (2.0 * p.D - p.C) / 3.0 * rs;
    }
}

__global__ void lda_kernel(int nspin, const double* __restrict__ rho, double* __restrict__ exc,
                           double* __restrict__ vxc, long long n) {
    const PZ U{-0.1423, 1.0529, 0.3334, 0.0311, -0.048, 0.0020, -0.0116};
    const PZ P{-0.0843, 1.3981, 0.2611, 0.01555, -0.0269, 0.0007, -0.0048};
    const double floor_ = 1e-14;
    const double cx = -0.75 * cbrt(3.0 / M_PI);
    const double fden = pow(2.0, 4.0 / 3.0) - 2.0;
    for (long long g = blockIdx.x * (long long)blockDim.x + threadIdx.x; g < n; g += (long long)gridDim.x * blockDim.x) {
        if (nspin == 1) {
            const double r = fmax(rho[g], floor_);
            const double ex = cx * cbrt(r);
            const double rs = cbrt(3.0 / (4.0 * M_PI * r));
            double ec, vc;
            pz_phase(rs, U, ec, vc);
            exc[g] = ex + ec;
            vxc[g] = 4.0 / 3.0 * ex + vc;
        } else {
            const double ru = rho[g], rd = rho[n + g];
            const double r = fmax(ru + rd, floor_);
            const double z = fmin(1.0, fmax(-1.0, (ru - rd) / r));
            const double exu = cx * cbrt(r);
            const double opz = 1.0 + z, omz = 1.0 - z;
            const double c_opz = cbrt(opz), c_omz = cbrt(omz);
            const double ex = exu * 0.5 * (opz * c_opz + omz * c_omz);
            const double rs = cbrt(3.0 / (4.0 * M_PI * r));
            double eu, mu_u, ep, mu_p;
            pz_phase(rs, U, eu, mu_u);
            pz_phase(rs, P, ep, mu_p);
            const double f = (opz * c_opz + omz * c_omz - 2.0) / fden;
            const double df = 4.0 / 3.0 * (c_opz - c_omz) / fden;
            const double ec = eu + f * (ep - eu);
            const double vcc = mu_u + f * (mu_p - mu_u);
            exc[g] = ex + ec;
            vxc[g] = 4.0 / 3.0 * exu * c_opz + vcc + (ep - eu) * df * (1.0 - z);
            vxc[n + g] = 4.0 / 3.0 * exu * c_omz + vcc + (ep - eu) * df * (-1.0 - z);
        }
    }
}

__global__ void veff_kernel(int nspin, const double* __restrict__ phi, const double* __restrict__ vxc,
                            double* __restrict__ veff, float* __restrict__ veff32, long long n) {
    for (long long g = blockIdx.x * (long long)blockDim.x + threadIdx.x; g < n; g += (long long)gridDim.x * blockDim.x)
        for (int s = 0; s < nspin; ++s) {
            const double v = phi[g] + vxc[s * n + g];
            veff[s * n + g] = v;
            veff32[s * n + g] = (float)v;
        }
}

// ---------------------------------------------------------------------------------------
// elementwise helpers
// ---------------------------------------------------------------------------------------
template <typename T>
__global__ void axpby_kernel(T* __restrict__ y, const T* __restrict__ x, T a, T b, long long n) {
    // y = a*x + b*y
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        y[i] = a * x[i] + b * y[i];
}
template <typename T, typename U>
__global__ void convert_add_kernel(T* __restrict__ y, const U* __restrict__ x, double a, double b, long long n) {
    // y = a*x + b*y with a type conversion (FP64 <-> FP32 vectors of the Poisson refinement)
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        y[i] = (T)(a * (double)x[i] + b * (double)y[i]);
}
__global__ void to_float_grid_kernel(const double* __restrict__ a, float* __restrict__ b, long long n) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        b[i] = (float)a[i];
}
__global__ void add_scalar_kernel(double* __restrict__ y, const double* __restrict__ s, double scale, long long n) {
    const double v = scale * s[0];
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        y[i] += v;
}

// Anderson history push: X[slot] = x - xprev, F[slot] = c*f - fprev; xprev = x, fprev = c*f
template <typename T>
__global__ void anderson_push_kernel(const T* __restrict__ x, const T* __restrict__ f, T c, T* __restrict__ xprev,
                                     T* __restrict__ fprev, T* __restrict__ Xs, T* __restrict__ Fs, int have_prev,
                                     long long n) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const T fi = c * f[i];
        if (have_prev) {
            Xs[i] = x[i] - xprev[i];
            Fs[i] = fi - fprev[i];
        }
        xprev[i] = x[i];
        fprev[i] = fi;
    }
}

// x += a*c*f - sum_j gamma_j (X_j + a F_j)   (gamma in device memory, m terms)
template <typename T>
__global__ void anderson_update_kernel(T* __restrict__ x, const T* __restrict__ f, T c, T a, const T* __restrict__ X,
                                       const T* __restrict__ F, const int* __restrict__ slots,
                                       const double* __restrict__ gamma, int m, long long n) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        T v = x[i] + a * c * f[i];
        for (int j = 0; j < m; ++j) {
            const long long o = (long long)slots[j] * n + i;
            v -= (T)gamma[j] * (X[o] + a * F[o]);
        }
        x[i] = v;
    }
}

// Sum each of ND per-thread values over the CTA into row[0..ND), with sh[ND][NW] of scratch.  32 values at a
// time are reduced together: at each of the five levels a lane keeps one half of its values and adds the partner
// lane's, so 31 additions serve 32 values where one shuffle tree per value takes 160 (FP64 additions are what such
// a reduction costs on this GPU).  The pairs added are the tree's (lane l with l + 16, then + 8, ...), so the sums
// are the same bit for bit.
template <int ND, int NW>
__device__ __forceinline__ void block_sum(const double* vals, double* __restrict__ row, double (*sh)[NW]) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int k0 = 0; k0 < ND; k0 += 32) {
        const int left = ND - k0;
        if (left >= 6) {   // fewer values: one tree each is as cheap
            double w[32];
#pragma unroll
            for (int k = 0; k < 32; ++k) w[k] = k < left ? vals[k0 + k < ND ? k0 + k : 0] : 0.0;
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) {
                const bool up = (lane & off) != 0;
#pragma unroll
                for (int k = 0; k < off; ++k) {
                    if (k < left) {   // values past ND are never kept
                        const double send = up ? w[k] : w[k + off];
                        const double keep = up ? w[k + off] : w[k];
                        w[k] = keep + __shfl_xor_sync(0xffffffffu, send, off);
                    }
                }
            }
            if (lane < left) sh[k0 + lane][warp] = w[0];
        } else {
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                if (k < left) {
                    double v = vals[k0 + k < ND ? k0 + k : 0];
                    for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
                    if (lane == 0) sh[k0 + k][warp] = v;
                }
            }
        }
    }
    __syncthreads();
    for (int k = threadIdx.x; k < ND; k += blockDim.x) {
        double v = 0.0;
        for (int w = 0; w < NW; ++w) v += sh[k][w];
        row[k] = v;
    }
}

// Gram of the history: G[i][j] = F_i . F_j (i <= j), r_i = F_i . (c f), plus f.f, for points
// [lo, hi) strided by `step`, summed over the CTA into row; C = history length at compile time keeps the
// accumulators in registers.
template <int C, int NW, typename T>
__device__ __forceinline__ void gram_accum(const T* __restrict__ F, const int* sl, const T* __restrict__ f, T c,
                                           long long n, long long lo, long long hi, long long step, double* row,
                                           double (*sh)[NW]) {
    constexpr int ND = C * (C + 1) / 2 + C + 1;
    T acc[ND];
#pragma unroll
    for (int k = 0; k < ND; ++k) acc[k] = T(0);
    for (long long i = lo; i < hi; i += step) {
        T v[C > 0 ? C : 1];
#pragma unroll
        for (int j = 0; j < C; ++j) v[j] = F[(long long)sl[j] * n + i];
        const T fi = c * f[i];
        int k = 0;
#pragma unroll
        for (int a = 0; a < C; ++a)
#pragma unroll
            for (int b = a; b < C; ++b) acc[k++] += v[a] * v[b];
#pragma unroll
        for (int a = 0; a < C; ++a) acc[k++] += v[a] * fi;
        acc[k] += fi * fi;
    }
    double out[ND];
#pragma unroll
    for (int k = 0; k < ND; ++k) out[k] = (double)acc[k];
    block_sum<ND, NW>(out, row, sh);
}

// the CTA's partial history Gram for a runtime history length m <= 16
template <int NW, typename T>
__device__ void gram_accum_dispatch(int m, const T* F, const int* sl, const T* f, T c, long long n, long long lo,
                                    long long hi, long long step, double* row, double (*sh)[NW]) {
    switch (m) {
#define SDFT_GRAM_CASE(CC) \
    case CC: gram_accum<CC, NW, T>(F, sl, f, c, n, lo, hi, step, row, sh); break;
        SDFT_GRAM_CASE(0) SDFT_GRAM_CASE(1) SDFT_GRAM_CASE(2) SDFT_GRAM_CASE(3) SDFT_GRAM_CASE(4) SDFT_GRAM_CASE(5)
        SDFT_GRAM_CASE(6) SDFT_GRAM_CASE(7) SDFT_GRAM_CASE(8) SDFT_GRAM_CASE(9) SDFT_GRAM_CASE(10) SDFT_GRAM_CASE(11)
        SDFT_GRAM_CASE(12) SDFT_GRAM_CASE(13) SDFT_GRAM_CASE(14) SDFT_GRAM_CASE(15) SDFT_GRAM_CASE(16)
#undef SDFT_GRAM_CASE
        default: break;
    }
}

constexpr int GRAM_MAXND = 16 * 17 / 2 + 16 + 1;

template <typename T>
__global__ void __launch_bounds__(RB) anderson_gram_kernel(const T* __restrict__ F, const int* __restrict__ slots,
                                                           int m, const T* __restrict__ f, T c, long long n,
                                                           double* __restrict__ part) {
    __shared__ double sh[GRAM_MAXND][RB / 32];
    int sl[16];
    for (int j = 0; j < m; ++j) sl[j] = slots[j];
    const long long step = (long long)gridDim.x * blockDim.x;
    const int nd = m * (m + 1) / 2 + m + 1;
    gram_accum_dispatch<RB / 32, T>(m, F, sl, f, c, n, blockIdx.x * (long long)blockDim.x + threadIdx.x, n, step,
                                    part + (long long)blockIdx.x * nd, sh);
}

// two at once: blockIdx.y 0 the history Gram with f, blockIdx.y 1 the norm of g
template <typename T>
__global__ void __launch_bounds__(RB) anderson_gram2_kernel(const T* __restrict__ F, const int* __restrict__ slots, int m,
                                                            const T* __restrict__ f, const T* __restrict__ g, T c,
                                                            long long n, double* __restrict__ part,
                                                            double* __restrict__ part_g) {
    __shared__ double sh[GRAM_MAXND][RB / 32];
    int sl[16];
    const int mm = blockIdx.y == 0 ? m : 0, nd = mm * (mm + 1) / 2 + mm + 1;
    for (int j = 0; j < mm; ++j) sl[j] = slots[j];
    gram_accum_dispatch<RB / 32, T>(mm, F, sl, blockIdx.y == 0 ? f : g, c, n,
                                    blockIdx.x * (long long)blockDim.x + threadIdx.x, n,
                                    (long long)gridDim.x * blockDim.x,
                                    (blockIdx.y == 0 ? part : part_g) + (long long)blockIdx.x * nd, sh);
}

// sum partials (one thread per entry, in block order), then solve (F^T F) gamma = F^T f by Gaussian elimination
// with partial pivoting in the first warp: the rows' factors by one lane each, then every (row, column) update by
// its own lane (one thread through a matrix in local memory took 25 us for m = 7, 14.7 us now)
__device__ void anderson_solve_block(const double* __restrict__ part, int nblk, int m, double* gamma, double* ff) {
    __shared__ double s[GRAM_MAXND];
    __shared__ double G[16][17], x[16];
    const int nd = m * (m + 1) / 2 + m + 1;
    for (int k = threadIdx.x; k < nd; k += blockDim.x) s[k] = ordered_sum<16>(part + k, nblk, nd);
    __syncthreads();
    if (threadIdx.x >= 32) return;
    const int lane = threadIdx.x;
    if (lane == 0) *ff = s[nd - 1];
    for (int e = lane; e < m * m; e += 32) {
        const int a = e / m, b = e - a * m, lo = min(a, b), hi = max(a, b);
        G[a][b] = s[lo * m - lo * (lo - 1) / 2 + hi - lo];
    }
    for (int a = lane; a < m; a += 32) G[a][m] = s[m * (m + 1) / 2 + a];
    __syncwarp();
    for (int col = 0; col < m; ++col) {
        int piv = col;
        for (int r = col + 1; r < m; ++r)
            if (fabs(G[r][col]) > fabs(G[piv][col])) piv = r;
        __syncwarp();
        if (piv != col && lane <= m) {
            const double t = G[col][lane];
            G[col][lane] = G[piv][lane];
            G[piv][lane] = t;
        }
        __syncwarp();
        const double d = G[col][col];
        const double fct = lane > col && lane < m && d != 0.0 ? G[lane][col] / d : 0.0;   // row `lane`
        __syncwarp();
        const int w = m + 1 - col, rows = m - 1 - col;
        for (int e0 = 0; e0 < rows * w; e0 += 32) {
            const int e = e0 + lane, i = e / w, q = col + e - i * w, r = col + 1 + i;
            const double f = __shfl_sync(0xffffffffu, fct, r & 31);
            if (e < rows * w) G[r][q] -= f * G[col][q];
        }
        __syncwarp();
    }
    // back substitution, row by row; a row subtracts its known terms in ascending column order
    for (int r = m - 1; r >= 0; --r) {
        if (lane == 0) {
            double v = G[r][m];
            for (int q = r + 1; q < m; ++q) v -= G[r][q] * x[q];
            x[r] = G[r][r] != 0.0 ? v / G[r][r] : 0.0;
        }
    }
    __syncwarp();
    if (lane < m) gamma[lane] = x[lane];
}

__global__ void anderson_solve_kernel(const double* __restrict__ part, int nblk, int m, double* __restrict__ gamma,
                                      double* __restrict__ ff) {
    anderson_solve_block(part, nblk, m, gamma, ff);
}

// blockIdx.x 0: solve the history Gram in part; 1: sum the norm's partials into *rr
__global__ void anderson_solve2_kernel(const double* __restrict__ part, const double* __restrict__ part_g, int nblk,
                                       int m, double* __restrict__ gamma, double* __restrict__ ff,
                                       double* __restrict__ rr) {
    if (blockIdx.x == 0) anderson_solve_block(part, nblk, m, gamma, ff);
    else anderson_solve_block(part_g, nblk, 0, nullptr, rr);
}

// ---------------------------------------------------------------------------------------
// density from orbitals (Eq. 2): rho[g] += weight * sum_n occ[n] |X[g,n]|^2 / dV
// ---------------------------------------------------------------------------------------
template <int KIND>  // 0 FP64 real, 1 FP64 complex, 2 FP32 paired real, 3 FP32 complex
__global__ void density_kernel(const void* __restrict__ X, const double* __restrict__ occ, int ncol, double scale,
                               long long ng, double* __restrict__ rho) {
    // states past the last one with |occ| > 1e-14 change rho below FP64 rounding and are not read;
    // the FP32 kinds square and weight in FP32 (the orbitals carry FP32 rounding already) and add
    // groups of eight pairs into the FP64 sum, so that the few FP64 pipes of the GPU do not bound
    // a pass that should stream the block at HBM speed
    extern __shared__ float occf[];
    __shared__ int nlast;
    if (threadIdx.x == 0) nlast = 0;
    __syncthreads();
    for (int n = threadIdx.x; n < ncol; n += blockDim.x) {
        const double o = occ[n];
        if (KIND >= 2) occf[n] = (float)o;
        if (fabs(o) > 1e-14) atomicMax(&nlast, n + 1);
    }
    __syncthreads();
    const int nc = nlast;
    for (long long g = blockIdx.x * (long long)blockDim.x + threadIdx.x; g < ng; g += (long long)gridDim.x * blockDim.x) {
        double s = 0.0;
        if (KIND == 0) {
            const double* x = (const double*)X;
            for (int n = 0; n < nc; ++n) {
                const double v = x[(long long)n * ng + g];
                s += occ[n] * v * v;
            }
        } else if (KIND == 1) {
            const double2* x = (const double2*)X;
            for (int n = 0; n < nc; ++n) {
                const double2 v = x[(long long)n * ng + g];
                s += occ[n] * (v.x * v.x + v.y * v.y);
            }
        } else if (KIND == 2) {
            const float2* x = (const float2*)X;
            const int np = (nc + 1) / 2;
            for (int p0 = 0; p0 < np; p0 += 8) {
                float sf = 0.f;
                if (p0 + 8 <= np) {   // eight loads in flight
                    float2 v[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i) v[i] = x[(long long)(p0 + i) * ng + g];
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        sf = fmaf(occf[2 * (p0 + i)], v[i].x * v[i].x, sf);
                        sf = fmaf(occf[2 * (p0 + i) + 1], v[i].y * v[i].y, sf);
                    }
                } else {
                    for (int p = p0; p < np; ++p) {
                        const float2 v = x[(long long)p * ng + g];
                        sf = fmaf(occf[2 * p], v.x * v.x, sf);
                        sf = fmaf(occf[2 * p + 1], v.y * v.y, sf);
                    }
                }
                s += (double)sf;
            }
        } else {
            const float2* x = (const float2*)X;
            for (int n0 = 0; n0 < nc; n0 += 8) {
                float sf = 0.f;
                const int n1 = min(nc, n0 + 8);
                for (int n = n0; n < n1; ++n) {
                    const float2 v = x[(long long)n * ng + g];
                    sf = fmaf(occf[n], v.x * v.x + v.y * v.y, sf);
                }
                s += (double)sf;
            }
        }
        rho[g] += scale * s;
    }
}

// ---------------------------------------------------------------------------------------
// Fermi level: bisection on sum_{s,k} w_k sum_n g = N_e, g = f_s / (1 + exp((e - mu)/kT))
// one CTA; writes occ, out[0] = mu, out[1] = -TS, out[2] = band energy sum w g e
// ---------------------------------------------------------------------------------------
__global__ void fermi_kernel(const double* __restrict__ eig, const double* __restrict__ kw, int nspin, int nk, int ns,
                             double nelec, double kT, double fs, double* __restrict__ occ, double* __restrict__ out) {
    __shared__ double red[1024 / 32];
    __shared__ double lo_s, hi_s;
    const int total = nspin * nk * ns;
    double emin = 1e300, emax = -1e300;
    for (int i = threadIdx.x; i < total; i += blockDim.x) {
        emin = fmin(emin, eig[i]);
        emax = fmax(emax, eig[i]);
    }
    auto block_reduce = [&](double v, int op) -> double {  // op 0 sum, 1 min, 2 max
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        for (int off = 16; off > 0; off >>= 1) {
            const double o = __shfl_down_sync(0xffffffffu, v, off);
            v = op == 0 ? v + o : (op == 1 ? fmin(v, o) : fmax(v, o));
        }
        __syncthreads();
        if (lane == 0) red[warp] = v;
        __syncthreads();
        double r = red[0];
        for (int w = 1; w < (int)(blockDim.x >> 5); ++w)
            r = op == 0 ? r + red[w] : (op == 1 ? fmin(r, red[w]) : fmax(r, red[w]));
        return r;
    };
    emin = block_reduce(emin, 1);
    emax = block_reduce(emax, 2);
    if (threadIdx.x == 0) {
        lo_s = emin - 50.0 * kT - 1.0;
        hi_s = emax + 50.0 * kT + 1.0;
    }
    __syncthreads();
    // safeguarded Newton on N(mu) = N_e: the bracket [lo, hi] shrinks every step (bisection
    // semantics as in the definition), the next trial point is the Newton step when it falls
    // inside the bracket, else the midpoint
    __shared__ double mu_s, red2[1024 / 32];
    __shared__ int done_s;
    if (threadIdx.x == 0) {
        mu_s = 0.5 * (lo_s + hi_s);
        done_s = 0;
    }
    __syncthreads();
    for (int it = 0; it < 200; ++it) {
        const double mid = mu_s;
        double cnt = 0.0, der = 0.0;
        for (int i = threadIdx.x; i < total; i += blockDim.x) {
            const int k = (i / ns) % nk;
            const double f = 0.5 * (1.0 - tanh(0.5 * (eig[i] - mid) / kT));
            cnt += kw[k] * fs * f;
            der += kw[k] * fs * f * (1.0 - f) / kT;
        }
        cnt = block_reduce(cnt, 0);
        {   // second sum through its own scratch row
            const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
            for (int off = 16; off > 0; off >>= 1) der += __shfl_down_sync(0xffffffffu, der, off);
            if (lane == 0) red2[warp] = der;
            __syncthreads();
            double r = red2[0];
            for (int w = 1; w < (int)(blockDim.x >> 5); ++w) r += red2[w];
            der = r;
        }
        if (threadIdx.x == 0) {
            if (cnt < nelec) lo_s = mid;
            else hi_s = mid;
            double next = 0.5 * (lo_s + hi_s);
            if (der > 0.0) {
                const double newton = mid + (nelec - cnt) / der;
                if (newton > lo_s && newton < hi_s) next = newton;
            }
            if (fabs(cnt - nelec) <= 1e-14 * fmax(1.0, nelec) || hi_s - lo_s < 1e-15 * fmax(1.0, fabs(mid))) {
                done_s = 1;
                next = mid;
            }
            mu_s = next;
        }
        __syncthreads();
        if (done_s) break;
    }
    const double mu = mu_s;
    double ts = 0.0, eb = 0.0;
    for (int i = threadIdx.x; i < total; i += blockDim.x) {
        const int k = (i / ns) % nk;
        const double g = fs * 0.5 * (1.0 - tanh(0.5 * (eig[i] - mu) / kT));
        occ[i] = g;
        const double f = g / fs;
        double t = 0.0;
        if (f > 0.0) t += f * log(f);
        if (f < 1.0) t += (1.0 - f) * log(1.0 - f);
        ts += kw[k] * fs * kT * t;
        eb += kw[k] * g * eig[i];
    }
    ts = block_reduce(ts, 0);
    eb = block_reduce(eb, 0);
    if (threadIdx.x == 0) {
        out[0] = mu;
        out[1] = ts;
        out[2] = eb;
    }
}

// ---------------------------------------------------------------------------------------
// forces
// ---------------------------------------------------------------------------------------
// Both parts are cut into chunks per atom (grid.y) whose partial sums go to part[atom][chunk][3] and are
// added in chunk order by force_finish_kernel: with one CTA per atom the 64-atom cell kept 64 of the 152
// SMs busy, each walking through all 154 columns one after another with two barriers and a redo of the
// projector's displacements and divisions per column (14.0 ms); the force of a chunk of columns reads the
// projector tables once for all of them and is bound by the FP64 pipe (4 fused multiply-adds per support
// point and column).  Measured on the 64-atom cell, 154 states: nonlocal part 14.0 -> 0.965 ms, local
// part 560 -> 375 us; two-atom cell, 8 states: 780 -> 37 us and 600 -> 34 us.
//
// local part of chunk blockIdx.y of atom blockIdx.x: sum_x (x - R - T)/r_loc^2 b_a(x - R - T) phi(x)
__global__ void __launch_bounds__(RB)
force_local_kernel(const AtomG* __restrict__ at, int n1, int n2, int n3, double h1, double h2, double h3,
                   const double* __restrict__ phi, double* __restrict__ part, int isolated) {
    const int a = blockIdx.x;
    const AtomG A = at[a];
    const double cut = A.cut_b;
    int lo[3], dim[3];
    const double h[3] = {h1, h2, h3};
    for (int d = 0; d < 3; ++d) {
        lo[d] = (int)ceil((A.pos[d] - cut) / h[d]);
        dim[d] = (int)floor((A.pos[d] + cut) / h[d]) - lo[d] + 1;
    }
    const int rows = dim[1] * dim[2];   // x-rows of the atom's box, one per warp at a time
    double acc[3] = {0, 0, 0};
    const double inv = 1.0 / (2.0 * A.w_b * A.w_b);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int row = blockIdx.y * (RB / 32) + warp; row < rows; row += gridDim.y * (RB / 32)) {
        const int iz = row / dim[1], iy = row - iz * dim[1];
        const int Iy = lo[1] + iy, Iz = lo[2] + iz;
        if (isolated && (Iy < 0 || Iy >= n2 || Iz < 0 || Iz >= n3)) continue;
        const double dy = Iy * h2 - A.pos[1], dz = Iz * h3 - A.pos[2];
        const double r2yz = dy * dy + dz * dz;
        if (r2yz > cut * cut) continue;
        const int g1 = ((Iy % n2) + n2) % n2, g2 = ((Iz % n3) + n3) % n3;
        const double* prow = phi + ((long long)g2 * n2 + g1) * n1;
        double sx = 0.0, s0 = 0.0;
        for (int ix = lane; ix < dim[0]; ix += 32) {
            const int Ix = lo[0] + ix;
            const double dx = Ix * h1 - A.pos[0];
            const double r2 = dx * dx + r2yz;
            if (r2 > cut * cut) continue;
            if (isolated && (Ix < 0 || Ix >= n1)) continue;
            const double s = exp(-r2 * inv) * prow[((Ix % n1) + n1) % n1];
            sx += dx * s;
            s0 += s;
        }
        acc[0] += sx;
        acc[1] += dy * s0;
        acc[2] += dz * s0;
    }
    const double f = A.amp_b / (A.w_b * A.w_b);
    __shared__ double sh[3][RB / 32];
    for (int d = 0; d < 3; ++d) {
        double v = acc[d];
        for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
        if (lane == 0) sh[d][warp] = v;
    }
    __syncthreads();
    if (threadIdx.x < 3) {
        double v = 0.0;
        for (int w = 0; w < RB / 32; ++w) v += sh[threadIdx.x][w];
        part[3 * ((long long)a * gridDim.y + blockIdx.y) + threadIdx.x] = f * v;
    }
}

// nonlocal part of columns [NC blockIdx.y, + NC) for atom blockIdx.x:
//   C_n = sum_j conj(beta_j) X[j,n], D_nd = sum_j conj(dbeta_j/dR_d) X[j,n],
//   part_d = sum_n g_n 2 Re(conj(C_n) D_nd); FP64 blocks (real or complex).
// A support point's weights (beta_j and beta_j disp_d / r_p^2) are formed once for the NC columns.
template <bool CPLX, int NC>
__global__ void __launch_bounds__(RB)
force_nl_kernel(const int* __restrict__ cnt, const int* __restrict__ idx, const int* __restrict__ img,
                const double* __restrict__ val, int cap, const double* __restrict__ X, int ncol, long long ng,
                const double* __restrict__ occ, const double* __restrict__ apos, const double* __restrict__ rp2,
                int n1, int n2, int n3, double h1, double h2, double h3, double* __restrict__ part) {
    constexpr int W = CPLX ? 2 : 1;   // doubles per value
    const int a = blockIdx.x;
    const int c0 = blockIdx.y * NC;
    const int m = cnt[a];
    const double R[3] = {apos[3 * a], apos[3 * a + 1], apos[3 * a + 2]};
    const double irp2 = 1.0 / rp2[a];
    double acc[NC][4][W];             // C, D_x, D_y, D_z per column
#pragma unroll
    for (int k = 0; k < NC; ++k)
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int w = 0; w < W; ++w) acc[k][q][w] = 0.0;
    for (int j = threadIdx.x; j < m; j += RB) {
        const long long e = (long long)a * cap + j;
        const int g = idx[e];
        double x[NC][W];
#pragma unroll
        for (int k = 0; k < NC; ++k) {
            const double* col = X + W * ((long long)min(c0 + k, ncol - 1) * ng + g);
#pragma unroll
            for (int w = 0; w < W; ++w) x[k][w] = col[w];
        }
        const int pk = img[e];
        const int t0 = (pk & 1023) - 512, t1 = ((pk >> 10) & 1023) - 512, t2 = ((pk >> 20) & 1023) - 512;
        const int gz = g / (n1 * n2), rem = g - gz * (n1 * n2), gy = rem / n1, gx = rem - gy * n1;
        // unwrapped box point I = g + t n;   displacement x_I - R
        double s[4];
        s[0] = 1.0;
        s[1] = ((gx + t0 * n1) * h1 - R[0]) * irp2;
        s[2] = ((gy + t1 * n2) * h2 - R[1]) * irp2;
        s[3] = ((gz + t2 * n3) * h3 - R[2]) * irp2;
        if constexpr (CPLX) {
            const double br = val[2 * e], bi = val[2 * e + 1];
#pragma unroll
            for (int k = 0; k < NC; ++k) {
                // conj(beta) * x
                const double pr = br * x[k][0] + bi * x[k][W - 1], pi = br * x[k][W - 1] - bi * x[k][0];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    acc[k][q][0] = fma(s[q], pr, acc[k][q][0]);
                    acc[k][q][W - 1] = fma(s[q], pi, acc[k][q][W - 1]);
                }
            }
        } else {
            const double b = val[e];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const double sb = q == 0 ? b : s[q] * b;
#pragma unroll
                for (int k = 0; k < NC; ++k) acc[k][q][0] = fma(sb, x[k][0], acc[k][q][0]);
            }
        }
    }
    __shared__ double sh[NC * 4 * W][RB / 32];
    __shared__ double tot[NC * 4 * W];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < NC; ++k)
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int w = 0; w < W; ++w) {
                double v = acc[k][q][w];
                for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
                if (lane == 0) sh[(k * 4 + q) * W + w][warp] = v;
            }
    __syncthreads();
    if (threadIdx.x < NC * 4 * W) {
        double v = 0.0;
        for (int w = 0; w < RB / 32; ++w) v += sh[threadIdx.x][w];
        tot[threadIdx.x] = v;
    }
    __syncthreads();
    if (threadIdx.x < 3) {
        const int q = threadIdx.x + 1;
        double f = 0.0;
        for (int k = 0; k < NC && c0 + k < ncol; ++k) {
            double p = tot[k * 4 * W] * tot[(k * 4 + q) * W];
            if (CPLX) p += tot[k * 4 * W + W - 1] * tot[(k * 4 + q) * W + W - 1];
            f += occ[c0 + k] * 2.0 * p;
        }
        part[3 * ((long long)a * gridDim.y + blockIdx.y) + threadIdx.x] = f;
    }
}

// F[3 a + d] -= scale (gamma[a]) sum_chunk part[a][chunk][d]; one warp per atom and component
__global__ void force_finish_kernel(const double* __restrict__ part, int nchunk, double scale,
                                    const double* __restrict__ gamma, double* __restrict__ F) {
    const int a = blockIdx.x, d = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double v = 0.0;
    for (int k = lane; k < nchunk; k += 32) v += part[3 * ((long long)a * nchunk + k) + d];
    for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
    if (lane == 0) F[3 * a + d] -= scale * (gamma ? gamma[a] : 1.0) * v;
}

inline unsigned nblocks(long long n, int bs = 256) {
    return (unsigned)std::min<long long>((n + bs - 1) / bs, 152LL * 16);
}

std::vector<AtomG> atom_g(sdft_ctx* c) {
    std::vector<AtomG> at(c->natom);
    for (int a = 0; a < c->natom; ++a) {
        const sdft_pseudo& s = c->species[c->types[a]];
        for (int d = 0; d < 3; ++d) at[a].pos[d] = c->pos[3 * a + d];
        at[a].amp_b = -s.Z * std::pow(2.0 * M_PI * s.r_loc * s.r_loc, -1.5);
        at[a].w_b = s.r_loc;
        at[a].cut_b = 10.0 * s.r_loc;
    }
    return at;
}

}  // namespace

// out[k] = a_k . b_k for k < count (<= 8), synchronously to host
void dots_host(sdft_ctx* c, int count, const double* const* a, const double* const* b, long long n, double* host_out) {
    SDFT_REQUIRE(count >= 1 && count <= 8, SDFT_ERR_INVALID_ARG, "dots_host: count");
    DotArgs P{};
    for (int k = 0; k < count; ++k) {
        P.a[k] = a[k];
        P.b[k] = b[k];
    }
    double* part = c->scal + 2048;
    double* out = c->scal + 1536;
    const int nblk = 128;  // 128 blocks x 8 dots fits in the 2048-double partial area
    auto launch = [&](auto kfn) { kfn<<<nblk, RB, 0, c->stream>>>(P, n, part); };
    switch (count) {
        case 1: launch(multidot_kernel<1>); break;
        case 2: launch(multidot_kernel<2>); break;
        case 3: launch(multidot_kernel<3>); break;
        case 4: launch(multidot_kernel<4>); break;
        case 5: launch(multidot_kernel<5>); break;
        case 6: launch(multidot_kernel<6>); break;
        case 7: launch(multidot_kernel<7>); break;
        default: launch(multidot_kernel<8>); break;
    }
    multidot_finish_kernel<<<1, 32, 0, c->stream>>>(part, nblk, count, out);
    SDFT_CUDA(cudaGetLastError());
    count_launch(c, 2);
    SDFT_CUDA(cudaMemcpyAsync(c->hscal, out, sizeof(double) * count, cudaMemcpyDeviceToHost, c->stream));
    SDFT_CUDA(cudaStreamSynchronize(c->stream));
    for (int k = 0; k < count; ++k) host_out[k] = c->hscal[k];
}

// ---------------------------------------------------------------------------------------
// PBE GGA, spin-unpolarized (paper Sec. 2.2 functionalities; Perdew, Burke & Ernzerhof 1996 with the
// Perdew-Wang 1992 correlation of the uniform gas).  On the grid: g_d = D_d rho with the order-12
// centred first-derivative stencil (periodic), sigma = sum_d g_d^2, f(rho, sigma) = rho eps_xc, and
// v_xc = f_rho - 2 sum_d D_d (f_sigma g_d), the exact derivative of E_xc = dV sum_g f (D_d^T = -D_d).
// ---------------------------------------------------------------------------------------
namespace {
struct D1Coef {
    double c[3][FD_RADIUS + 1];   // c_k / h_d, k = 1..6: (D_d u)(x) = sum_k c_k (u(x + k e_d) - u(x - k e_d))
};

// out_d = D_d u for the three axes (in0 == in1 == in2 == u), or out0 -= sum_d D_d in_d (accumulate)
template <bool DIV>
__global__ void __launch_bounds__(256) d1_kernel(const double* __restrict__ in0, const double* __restrict__ in1,
                                                 const double* __restrict__ in2, double* __restrict__ out0,
                                                 double* __restrict__ out1, double* __restrict__ out2, D1Coef K,
                                                 int n1, int n2, int n3) {
    const int plane = n1 * n2;
    const int ng = plane * n3;
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= ng) return;
    const int k = g / plane;
    const int rem = g - k * plane;
    const int j = rem / n1;
    const int i = rem - j * n1;
    const int row = g - i, col = g - j * n1, pl = g - k * plane;
    double dx = 0.0, dy = 0.0, dz = 0.0;
#pragma unroll
    for (int r = 1; r <= FD_RADIUS; ++r) {
        int ip = i + r, im = i - r, jp = j + r, jm = j - r, kp = k + r, km = k - r;
        ip -= ip >= n1 ? n1 : 0;
        im += im < 0 ? n1 : 0;
        jp -= jp >= n2 ? n2 : 0;
        jm += jm < 0 ? n2 : 0;
        kp -= kp >= n3 ? n3 : 0;
        km += km < 0 ? n3 : 0;
        dx += K.c[0][r] * (in0[row + ip] - in0[row + im]);
        dy += K.c[1][r] * (in1[col + jp * n1] - in1[col + jm * n1]);
        dz += K.c[2][r] * (in2[pl + kp * plane] - in2[pl + km * plane]);
    }
    if (DIV) {
        out0[g] -= dx + dy + dz;
    } else {
        out0[g] = dx;
        out1[g] = dy;
        out2[g] = dz;
    }
}

constexpr double PBE_KAPPA = 0.804;
constexpr double PBE_BETA = 0.06672455060314922;
constexpr double PW92_A = 0.031091, PW92_A1 = 0.21370, PW92_B1 = 7.5957, PW92_B2 = 3.5876, PW92_B3 = 1.6382,
                 PW92_B4 = 0.49294;

// eps_xc (per electron), f_rho and f_sigma of PBE at one point, analytic derivatives
__device__ void pbe_eval(double rho, double sigma, double& eps, double& frho, double& fsig) {
    const double pi = 3.14159265358979323846;
    const double mu = PBE_BETA * pi * pi / 3.0;
    const double gam = (1.0 - log(2.0)) / (pi * pi);
    const double r = fmax(rho, 1e-14);
    const double kf = cbrt(3.0 * pi * pi * r);
    const double exu = -3.0 * kf / (4.0 * pi);
    // exchange: f_x = r exu F_x(s2), s2 = sigma / (4 kf^2 r^2) ~ sigma r^(-8/3)
    const double s2den = 4.0 * kf * kf * r * r;
    const double s2 = sigma / s2den;
    const double den = PBE_KAPPA + mu * s2;
    const double Fx = 1.0 + PBE_KAPPA - PBE_KAPPA * PBE_KAPPA / den;
    const double dFx = mu * PBE_KAPPA * PBE_KAPPA / (den * den);   // dF_x / ds2
    const double fx = r * exu * Fx;
    const double fx_r = (4.0 / 3.0) * exu * Fx - (8.0 / 3.0) * exu * dFx * s2;
    const double fx_s = r * exu * dFx / s2den;
    // PW92 correlation of the uniform gas, eps_c(rs), rs = (3 / (4 pi r))^(1/3)
    const double rs = cbrt(3.0 / (4.0 * pi * r));
    const double sq = sqrt(rs);
    const double Q = 2.0 * PW92_A * (PW92_B1 * sq + PW92_B2 * rs + PW92_B3 * rs * sq + PW92_B4 * rs * rs);
    const double dQ = 2.0 * PW92_A * (0.5 * PW92_B1 / sq + PW92_B2 + 1.5 * PW92_B3 * sq + 2.0 * PW92_B4 * rs);
    const double Lq = log1p(1.0 / Q);
    const double ec = -2.0 * PW92_A * (1.0 + PW92_A1 * rs) * Lq;
    const double dec_drs = -2.0 * PW92_A * PW92_A1 * Lq + 2.0 * PW92_A * (1.0 + PW92_A1 * rs) * dQ / (Q * (1.0 + Q));
    const double dec_dr = -dec_drs * rs / (3.0 * r);
    // gradient correction H(ec, t2), t2 = sigma / (4 ks^2 r^2) ~ sigma r^(-7/3), ks^2 = 4 kf / pi
    const double t2den = 16.0 * kf * r * r / pi;
    const double t2 = sigma / t2den;
    const double E = exp(-ec / gam);
    const double A = (PBE_BETA / gam) / (E - 1.0);
    const double dA_dec = (PBE_BETA / (gam * gam)) * E / ((E - 1.0) * (E - 1.0));
    const double y = A * t2;
    const double Dn = 1.0 + y + y * y;
    const double Z = (PBE_BETA / gam) * t2 * (1.0 + y) / Dn;
    const double H = gam * log1p(Z);
    const double dH_dt2 = PBE_BETA * (1.0 + 2.0 * y) / ((1.0 + Z) * Dn * Dn);
    const double dH_dA = -PBE_BETA * t2 * t2 * y * (2.0 + y) / ((1.0 + Z) * Dn * Dn);
    const double fc = r * (ec + H);
    const double fc_r = ec + H + r * dec_dr * (1.0 + dH_dA * dA_dec) - (7.0 / 3.0) * dH_dt2 * t2;
    const double fc_s = r * dH_dt2 / t2den;
    eps = (fx + fc) / r;
    frho = fx_r + fc_r;
    fsig = fx_s + fc_s;
}

// exc = eps_xc, vxc = f_rho, w_d = 2 f_sigma g_d  (the divergence kernel then subtracts sum_d D_d w_d)
__global__ void pbe_point_kernel(const double* __restrict__ rho, const double* __restrict__ g0,
                                 const double* __restrict__ g1, const double* __restrict__ g2,
                                 double* __restrict__ exc, double* __restrict__ vxc, double* __restrict__ w0,
                                 double* __restrict__ w1, double* __restrict__ w2, long long n) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const double a = g0[i], b = g1[i], cc = g2[i];
        double eps, fr, fs;
        pbe_eval(rho[i], a * a + b * b + cc * cc, eps, fr, fs);
        exc[i] = eps;
        vxc[i] = fr;
        w0[i] = 2.0 * fs * a;
        w1[i] = 2.0 * fs * b;
        w2[i] = 2.0 * fs * cc;
    }
}
}  // namespace

static void gga_pbe_device(sdft_ctx* c, const double* rho, double* exc, double* vxc) {
    const long long n = c->ng;
    if (!c->gga_ws) c->gga_ws = (double*)ctx_alloc(c, sizeof(double) * 6 * (size_t)n);
    double* g = c->gga_ws;
    double* w = c->gga_ws + 3 * n;
    // first-derivative weights c_k = (-1)^(k+1) (p!)^2 / (k (p-k)! (p+k)!), p = 6
    D1Coef K;
    {
        auto fact = [](int m) {
            double f = 1.0;
            for (int q = 2; q <= m; ++q) f *= q;
            return f;
        };
        const int p = FD_RADIUS;
        for (int d = 0; d < 3; ++d) {
            K.c[d][0] = 0.0;
            for (int k = 1; k <= p; ++k)
                K.c[d][k] = ((k % 2) ? 1.0 : -1.0) * fact(p) * fact(p) / (k * fact(p - k) * fact(p + k)) / c->h[d];
        }
    }
    const unsigned nbk = (unsigned)((n + 255) / 256);
    d1_kernel<false><<<nbk, 256, 0, c->stream>>>(rho, rho, rho, g, g + n, g + 2 * n, K, c->n[0], c->n[1], c->n[2]);
    pbe_point_kernel<<<nblocks(n), 256, 0, c->stream>>>(rho, g, g + n, g + 2 * n, exc, vxc, w, w + n, w + 2 * n, n);
    d1_kernel<true><<<nbk, 256, 0, c->stream>>>(w, w + n, w + 2 * n, vxc, nullptr, nullptr, K, c->n[0], c->n[1],
                                                 c->n[2]);
    SDFT_CUDA(cudaGetLastError());
    count_launch(c, 3);
}

void lda_device(sdft_ctx* c, int nspin, const double* rho, double* exc, double* vxc, size_t n) {
    if (c->opt.xc == SDFT_XC_GGA_PBE) {
        SDFT_REQUIRE(nspin == 1 && (long long)n == c->ng, SDFT_ERR_INVALID_ARG,
                     "PBE: spin-unpolarized densities on the context's grid only");
        gga_pbe_device(c, rho, exc, vxc);
        return;
    }
    lda_kernel<<<nblocks((long long)n), 256, 0, c->stream>>>(nspin, rho, exc, vxc, (long long)n);
    SDFT_CUDA(cudaGetLastError());
    count_launch(c);
}

// V_eff^s = phi + v_xc^s from rho_in (Poisson solved by the caller into c->phi)
void veff_assemble(sdft_ctx* c) {
    const int ns = c->opt.nspin;
    double* vxc = c->work64 + 2 * c->ng;  // [nspin][ng]
    lda_device(c, ns, c->rho_in, c->exc, vxc, (size_t)c->ng);
    veff_kernel<<<nblocks(c->ng), 256, 0, c->stream>>>(ns, c->phi, vxc, c->veff, c->veff32, c->ng);
    SDFT_CUDA(cudaGetLastError());
    count_launch(c);
}

void veff_to_float(sdft_ctx* c, int spin) {
    const long long n = c->ng;
    to_float_grid_kernel<<<nblocks(n), 256, 0, c->stream>>>(c->veff + spin * n, c->veff32 + spin * n, n);
    SDFT_CUDA(cudaGetLastError());
    count_launch(c);
}

// ---------------------------------------------------------------------------------------
// Single-vector Laplacian step for the Poisson solver: out = -2 alpha (-1/2 L x) - beta b, i.e.
// with alpha = -2, beta = -1:  out = b + L x (the residual of -L x = b).  One thread per grid
// point with direct neighbour loads: the vector is a few MB and stays in L2, so a flat grid of
// short independent threads beats the z-marching tile kernel built for orbital blocks.
// ---------------------------------------------------------------------------------------
template <typename T>
struct LapCoefT {        // in the vector's own type: converting on use would cost an FP64-rate instruction each
    T c[3][FD_RADIUS + 1];  // -1/2 w_r / h_d^2
    T c0;
};
using LapCoef = LapCoefT<double>;
template <typename T>
LapCoefT<T> lap_coef(const sdft_ctx* c) {
    LapCoefT<T> K;
    for (int r = 0; r <= FD_RADIUS; ++r) {
        K.c[0][r] = (T)c->coef.cx[r];
        K.c[1][r] = (T)c->coef.cy[r];
        K.c[2][r] = (T)c->coef.cz[r];
    }
    K.c0 = (T)c->coef.c0;
    return K;
}

__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }

template <typename T, bool DIR>
__device__ __forceinline__ T laplacian_residual_at(const T* __restrict__ x, const T* __restrict__ b, const LapCoefT<T>& K,
                                                   int n1, int n2, int n3, T shift, int g) {
    // 32-bit indices: the grid has < 2^31 points
    const int plane = n1 * n2;
    const int k = g / plane;
    const int rem = g - k * plane;
    const int j = rem / n1;
    const int i = rem - j * n1;
    const int row = g - i, col = g - j * n1, pl = g - k * plane;
    T acc = mul_rn(K.c0, x[g]);   // roundings spelled out: a contraction of the first terms would change the sum
#pragma unroll
    for (int r = 1; r <= FD_RADIUS; ++r) {
        int ip = i + r, im = i - r, jp = j + r, jm = j - r, kp = k + r, km = k - r;
        ip -= ip >= n1 ? n1 : 0;
        im += im < 0 ? n1 : 0;
        jp -= jp >= n2 ? n2 : 0;
        jm += jm < 0 ? n2 : 0;
        kp -= kp >= n3 ? n3 : 0;
        km += km < 0 ? n3 : 0;
        if (DIR) {   // zero beyond the grid (isolated systems: ghost values enter through b)
            acc = fma(K.c[0][r], (i + r < n1 ? x[row + ip] : (T)0) + (i - r >= 0 ? x[row + im] : (T)0), acc);
            acc = fma(K.c[1][r], (j + r < n2 ? x[col + jp * n1] : (T)0) + (j - r >= 0 ? x[col + jm * n1] : (T)0), acc);
            acc = fma(K.c[2][r], (k + r < n3 ? x[pl + kp * plane] : (T)0) + (k - r >= 0 ? x[pl + km * plane] : (T)0), acc);
        } else {
            acc = fma(K.c[0][r], x[row + ip] + x[row + im], acc);
            acc = fma(K.c[1][r], x[col + jp * n1] + x[col + jm * n1], acc);
            acc = fma(K.c[2][r], x[pl + kp * plane] + x[pl + km * plane], acc);
        }
    }
    // -L x = 2 * (-1/2 L x): b + L x - shift x = b - 2 acc - shift x  (residual of (-L + shift) x = b)
    return fma(-shift, x[g], fma((T)-2, acc, b[g]));
}

template <typename T, bool DIR>
__global__ void __launch_bounds__(256) laplacian_residual_kernel(const T* __restrict__ x, const T* __restrict__ b,
                                                                 T* __restrict__ out,
                                                                 const __grid_constant__ LapCoefT<T> K, int n1, int n2,
                                                                 int n3, T shift) {
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g < n1 * n2 * n3) out[g] = laplacian_residual_at<T, DIR>(x, b, K, n1, n2, n3, shift, g);
}

template <typename T>
void laplacian_residual(sdft_ctx* c, const T* x, const T* b, T* out, T shift = T(0)) {
    const LapCoefT<T> K = lap_coef<T>(c);
    auto launch = [&](auto kfn) {
        kfn<<<(unsigned)((c->ng + 255) / 256), 256, 0, c->stream>>>(x, b, out, K, c->n[0], c->n[1], c->n[2], shift);
    };
    if (c->opt.boundary == SDFT_BC_DIRICHLET) launch(laplacian_residual_kernel<T, true>);
    else launch(laplacian_residual_kernel<T, false>);
    SDFT_CUDA(cudaGetLastError());
    count_launch(c);
}

// One FP64 AAR iteration but for the Anderson step, in one launch: r = residual of x, the history push with
// f = c r (anderson_push_kernel), and either the Richardson step into the other x buffer, xn = omega c r + x, or
// (xn null, an Anderson step follows) r itself.  Separate kernels for these read x, r and the previous iterate
// again and cost two more launches per iteration (two-atom cell, 24^3: 4.8 + 1.9 + 1.7 us -> 4.1 us).
template <bool DIR>
__global__ void __launch_bounds__(256)
aar_step_kernel(const double* __restrict__ x, const double* __restrict__ b, double* __restrict__ r_out,
                double* __restrict__ xn, double* __restrict__ xprev, double* __restrict__ fprev, double* __restrict__ Xs,
                double* __restrict__ Fs, const __grid_constant__ LapCoef K, int n1, int n2, int n3, double shift,
                double cj, double wcj, int have_prev) {
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= n1 * n2 * n3) return;
    const double r = laplacian_residual_at<double, DIR>(x, b, K, n1, n2, n3, shift, g);
    const double xg = x[g];
    if (have_prev) {
        Xs[g] = xg - xprev[g];
        Fs[g] = __dsub_rn(__dmul_rn(cj, r), fprev[g]);
    }
    xprev[g] = xg;
    fprev[g] = cj * r;
    if (xn) xn[g] = fma(wcj, r, xg);
    else r_out[g] = r;
}

void aar_step(sdft_ctx* c, const double* x, const double* b, double* r, double* xn, double* xprev, double* fprev,
              double* Xs, double* Fs, double shift, double cj, double omega, bool have_prev) {
    const LapCoef K = lap_coef<double>(c);
    // small grids: CTAs small enough that every SM's (few) FP64 pipes get one
    const int bs = (int)std::min<long long>(256, (c->ng + 152 * 32 - 1) / (152 * 32) * 32);
    auto launch = [&](auto kfn) {
        kfn<<<(unsigned)((c->ng + bs - 1) / bs), bs, 0, c->stream>>>(x, b, r, xn, xprev, fprev, Xs, Fs, K, c->n[0],
                                                                    c->n[1], c->n[2], shift, cj, omega * cj, have_prev);
    };
    if (c->opt.boundary == SDFT_BC_DIRICHLET) launch(aar_step_kernel<true>);
    else launch(aar_step_kernel<false>);
    SDFT_CUDA(cudaGetLastError());
    count_launch(c);
}

// ---------------------------------------------------------------------------------------
// Isolated systems (paper Sec. 2, 2.1: Dirichlet boundary conditions with multipole boundary values).
// q_lm = dV sum_g f_g r^l Y_lm about the centre of the grid box (l <= 6, real orthonormal Y_lm), and in
// the 6 ghost layers phi = sum 4 pi / (2l + 1) q_lm Y_lm / r^(l+1); inside -L0 phi = 4 pi f + G with
// L0 the zero-padded Laplacian and G the ghost values' share of the stencil.
// ---------------------------------------------------------------------------------------
namespace {
constexpr int MP_LMAX = 6, MP_NLM = (MP_LMAX + 1) * (MP_LMAX + 1);

// real orthonormal spherical harmonics of the direction (x, y, z), index l^2 + l + m (associated Legendre
// functions by the standard three-term recurrence; any real orthonormal basis gives the same potential)
__device__ void real_sh(double x, double y, double z, double* Y) {
    const double r = sqrt(x * x + y * y + z * z);
    double ct = 1.0, st = 0.0, cp = 1.0, sp = 0.0;
    if (r > 0.0) {
        ct = z / r;
        const double rxy = sqrt(x * x + y * y);
        st = rxy / r;
        if (rxy > 0.0) {
            cp = x / rxy;
            sp = y / rxy;
        }
    }
    double P[MP_LMAX + 1][MP_LMAX + 1];
    P[0][0] = 1.0;
    for (int m = 1; m <= MP_LMAX; ++m) P[m][m] = P[m - 1][m - 1] * (2 * m - 1) * st;
    for (int m = 0; m < MP_LMAX; ++m) P[m + 1][m] = ct * (2 * m + 1) * P[m][m];
    for (int m = 0; m <= MP_LMAX; ++m)
        for (int l = m + 2; l <= MP_LMAX; ++l)
            P[l][m] = ((2 * l - 1) * ct * P[l - 1][m] - (l + m - 1) * P[l - 2][m]) / (l - m);
    double cm[MP_LMAX + 1], sm[MP_LMAX + 1];
    cm[0] = 1.0;
    sm[0] = 0.0;
    for (int m = 1; m <= MP_LMAX; ++m) {
        cm[m] = cm[m - 1] * cp - sm[m - 1] * sp;
        sm[m] = sm[m - 1] * cp + cm[m - 1] * sp;
    }
    for (int l = 0; l <= MP_LMAX; ++l) {
        double ratio = 1.0;   // (l - m)! / (l + m)!
        for (int m = 0; m <= l; ++m) {
            if (m > 0) ratio /= (double)((l + m) * (l - m + 1));
            const double N = sqrt((2 * l + 1) / (4.0 * 3.14159265358979323846) * ratio);
            if (m == 0) {
                Y[l * l + l] = N * P[l][0];
            } else {
                Y[l * l + l + m] = 1.4142135623730951 * N * P[l][m] * cm[m];
                Y[l * l + l - m] = 1.4142135623730951 * N * P[l][m] * sm[m];
            }
        }
    }
}

// per-block partial moments part[block][lm] of f about the centre (c0, c1, c2)
__global__ void __launch_bounds__(256) multipole_kernel(const double* __restrict__ f, int n1, int n2, int n3,
                                                        double h1, double h2, double h3, double c0, double c1,
                                                        double c2, double* __restrict__ part) {
    __shared__ double sh[MP_NLM][8];
    double acc[MP_NLM];
    for (int k = 0; k < MP_NLM; ++k) acc[k] = 0.0;
    const long long ng = (long long)n1 * n2 * n3;
    for (long long g = blockIdx.x * (long long)blockDim.x + threadIdx.x; g < ng; g += (long long)gridDim.x * blockDim.x) {
        const int i = (int)(g % n1), j = (int)((g / n1) % n2), k = (int)(g / ((long long)n1 * n2));
        const double x = i * h1 - c0, y = j * h2 - c1, z = k * h3 - c2;
        const double r = sqrt(x * x + y * y + z * z);
        double Y[MP_NLM];
        real_sh(x, y, z, Y);
        double rl = f[g];
        for (int l = 0; l <= MP_LMAX; ++l) {
            for (int m = -l; m <= l; ++m) acc[l * l + l + m] += rl * Y[l * l + l + m];
            rl *= r;
        }
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int k = 0; k < MP_NLM; ++k) {
        double v = acc[k];
        for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
        if (lane == 0) sh[k][warp] = v;
    }
    __syncthreads();
    for (int k = threadIdx.x; k < MP_NLM; k += blockDim.x) {
        double v = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) v += sh[k][w];
        part[(long long)blockIdx.x * MP_NLM + k] = v;
    }
}

__device__ double multipole_phi(const double* q, double x, double y, double z) {
    double Y[MP_NLM];
    real_sh(x, y, z, Y);
    const double r = sqrt(x * x + y * y + z * z);
    const double ir = 1.0 / r;
    double irl = ir, v = 0.0;   // r^-(l+1)
    for (int l = 0; l <= MP_LMAX; ++l) {
        double s = 0.0;
        for (int m = -l; m <= l; ++m) s += q[l * l + l + m] * Y[l * l + l + m];
        v += 4.0 * 3.14159265358979323846 / (2 * l + 1) * s * irl;
        irl *= ir;
    }
    return v;
}

// rhs = 4 pi f + G, G = sum over stencil neighbours beyond the grid of (w_r / h_d^2) phi_ghost
// (K.c = -1/2 w_r / h_d^2, so G = -2 sum K.c phi_ghost)
__global__ void __launch_bounds__(256) dirichlet_rhs_kernel(const double* __restrict__ f, double* __restrict__ rhs,
                                                            const double* __restrict__ q, LapCoef K, int n1, int n2,
                                                            int n3, double h1, double h2, double h3, double c0,
                                                            double c1, double c2) {
    const long long ng = (long long)n1 * n2 * n3;
    for (long long g = blockIdx.x * (long long)blockDim.x + threadIdx.x; g < ng; g += (long long)gridDim.x * blockDim.x) {
        const int I[3] = {(int)(g % n1), (int)((g / n1) % n2), (int)(g / ((long long)n1 * n2))};
        const int n[3] = {n1, n2, n3};
        const double h[3] = {h1, h2, h3}, cc[3] = {c0, c1, c2};
        double v = 4.0 * 3.14159265358979323846 * f[g];
        for (int d = 0; d < 3; ++d)
            for (int r = 1; r <= FD_RADIUS; ++r)
                for (int sgn = -1; sgn <= 1; sgn += 2) {
                    const int id = I[d] + sgn * r;
                    if (id >= 0 && id < n[d]) continue;
                    double X[3];
                    for (int e = 0; e < 3; ++e) X[e] = (e == d ? id : I[e]) * h[e] - cc[e];
                    v += -2.0 * K.c[d][r] * multipole_phi(q, X[0], X[1], X[2]);
                }
        rhs[g] = v;
    }
}
}  // namespace

// rhs of the isolated Poisson problem for charge f (device [ngrid])
static void isolated_poisson_rhs(sdft_ctx* c, const double* f, double* rhs) {
    const int nblk = 128;
    double* part = c->work64 + 27 * c->ng;   // nblk * 49 doubles (the grid's last scratch vector)
    SDFT_REQUIRE((long long)nblk * MP_NLM <= c->ng, SDFT_ERR_INVALID_ARG, "isolated Poisson: grid too small");
    double cen[3];
    for (int d = 0; d < 3; ++d) cen[d] = 0.5 * (c->n[d] - 1) * c->h[d];
    multipole_kernel<<<nblk, 256, 0, c->stream>>>(f, c->n[0], c->n[1], c->n[2], c->h[0], c->h[1], c->h[2], cen[0], cen[1],
                                                  cen[2], part);
    SDFT_CUDA(cudaGetLastError());
    count_launch(c);
    std::vector<double> hp((size_t)nblk * MP_NLM);
    SDFT_CUDA(cudaMemcpyAsync(hp.data(), part, sizeof(double) * hp.size(), cudaMemcpyDeviceToHost, c->stream));
    SDFT_CUDA(cudaStreamSynchronize(c->stream));
    double q[MP_NLM];
    for (int k = 0; k < MP_NLM; ++k) {
        double s = 0.0;
        for (int b = 0; b < nblk; ++b) s += hp[(size_t)b * MP_NLM + k];
        q[k] = c->dV * s;
    }
    double* dq = c->scal + 1700;   // [1700, 1749): multipole moments (free part of the scalar area)
    std::memcpy(c->hscal + 1700, q, sizeof(q));
    SDFT_CUDA(cudaMemcpyAsync(dq, c->hscal + 1700, sizeof(q), cudaMemcpyHostToDevice, c->stream));
    const LapCoef K = lap_coef<double>(c);
    dirichlet_rhs_kernel<<<nblocks(c->ng), 256, 0, c->stream>>>(f, rhs, dq, K, c->n[0], c->n[1], c->n[2], c->h[0],
                                                               c->h[1], c->h[2], cen[0], cen[1], cen[2]);
    SDFT_CUDA(cudaGetLastError());
    count_launch(c);
}

// ---------------------------------------------------------------------------------------
// AAR Poisson (Pratapa, Suryanarayana & Pask 2016; Suryanarayana et al. 2019):
// A = -L_h, Jacobi preconditioner, Richardson steps with omega, Anderson every p-th step.
// ---------------------------------------------------------------------------------------
namespace {
struct Event {   // without timing
    cudaEvent_t e = nullptr;
    Event() { SDFT_CUDA(cudaEventCreateWithFlags(&e, cudaEventDisableTiming)); }
    ~Event() { cudaEventDestroy(e); }
    Event(const Event&) = delete;
    Event& operator=(const Event&) = delete;
};
}  // namespace

int poisson_aar(sdft_ctx* c, const double* f, double* phi, double tol, int max_iter) {
    const long long n = c->ng;
    ScopedTimer timer(c, SDFT_K_POISSON);
    const double omega = 0.6, beta = 0.6;
    const int m = 7, p = 6;
    // workspace: rhs, r, xprev, fprev, X[m], F[m]
    double* rhs = c->work64 + 0 * n;
    double* r = c->work64 + 1 * n;
    double* xprev = c->work64 + 4 * n;
    double* fprev = c->work64 + 5 * n;
    double* hist = c->work64 + 6 * n;  // 2*m vectors
    double* Xs = hist;
    double* Fs = hist + (long long)m * n;
    double* gam = c->scal + 64;
    int* slots = (int*)(c->scal + 96);
    double* ffv = c->scal + 128;
    double* part = c->scal + 4096;
    const bool isolated = c->opt.boundary == SDFT_BC_DIRICHLET;
    // rhs = 4 pi (f - mean f); phi -= mean(phi)   (isolated: rhs = 4 pi f + ghost term, no gauge)
    if (isolated) {
        isolated_poisson_rhs(c, f, rhs);
    } else {
        double* ones = c->work64 + 3 * n;
        SDFT_CUDA(cudaMemsetAsync(ones, 0, sizeof(double) * n, c->stream));
        c->hscal[0] = 1.0;
        SDFT_CUDA(cudaMemcpyAsync(c->scal, c->hscal, sizeof(double), cudaMemcpyHostToDevice, c->stream));
        add_scalar_kernel<<<nblocks(n), 256, 0, c->stream>>>(ones, c->scal, 1.0, n);
        const double* A[2] = {f, phi};
        const double* B[2] = {ones, ones};
        double s[2];
        dots_host(c, 2, A, B, n, s);
        SDFT_CUDA(cudaMemcpyAsync(rhs, f, sizeof(double) * n, cudaMemcpyDeviceToDevice, c->stream));
        c->hscal[0] = -s[0] / n;
        c->hscal[1] = -s[1] / n;
        SDFT_CUDA(cudaMemcpyAsync(c->scal, c->hscal, 2 * sizeof(double), cudaMemcpyHostToDevice, c->stream));
        add_scalar_kernel<<<nblocks(n), 256, 0, c->stream>>>(rhs, c->scal, 1.0, n);
        add_scalar_kernel<<<nblocks(n), 256, 0, c->stream>>>(phi, c->scal + 1, 1.0, n);
        axpby_kernel<double><<<nblocks(n), 256, 0, c->stream>>>(rhs, rhs, 0.0, 4.0 * M_PI, n);
        SDFT_CUDA(cudaGetLastError());
        count_launch(c, 5);
    }
    double bnorm2;
    {
        const double* A[1] = {rhs};
        dots_host(c, 1, A, A, n, &bnorm2);
    }
    if (bnorm2 == 0.0) {
        SDFT_CUDA(cudaMemsetAsync(phi, 0, sizeof(double) * n, c->stream));
        return 0;
    }
    // Jacobi: diag(-L) = -(sum_d w0/h_d^2) = 2*c0 (c0 = -1/2 sum_d w0/h^2 > 0)
    const double cj = 1.0 / (2.0 * c->coef.c0);
    int count = 0, head = 0, it = 0;
    int hslots[16];
    // A Richardson step writes another buffer than it reads.  The residual of an Anderson step is read back while the
    // Richardson steps that would follow it run, not after it (five steps of 4 us; two-atom SCF 19.31 -> 19.14 ms);
    // they leave the Anderson iterate alone, which is the result if that residual is small enough.
    double* buf[3] = {phi, c->work64 + 2 * n, c->work64 + 3 * n};
    int cur = 0, keep = -1, asked = -1;      // buffer and iteration of the Anderson step whose residual is on its way
    Event read;
    auto converged = [&] {
        SDFT_CUDA(cudaEventSynchronize(read.e));
        asked = -1;
        const double rn2 = c->hscal[0] / (cj * cj);   // ||r||^2 = ffv / cj^2
        if (!std::isfinite(rn2)) {
            SDFT_CUDA(cudaStreamSynchronize(c->stream));   // nothing writes phi after the error is reported
            throw Error{SDFT_ERR_NONFINITE, "Poisson residual is not finite"};
        }
        return rn2 <= tol * tol * bnorm2;
    };
    for (it = 0; it < max_iter; ++it) {
        // r = rhs - A phi = rhs + L phi, history push with f = cj * r, and the Richardson step phi += omega cj r
        const int slot = head;
        if (it > 0) {
            head = (head + 1) % m;
            count = std::min(count + 1, m);
        }
        const bool anderson = ((it + 1) % p == 0) && count > 0;
        if (anderson && asked >= 0) {
            const int at = asked;
            if (converged()) {
                cur = keep;
                it = at + 1;
                break;
            }
            keep = -1;
        }
        int next = (cur + 1) % 3;
        if (next == keep) next = (cur + 2) % 3;
        aar_step(c, buf[cur], rhs, r, anderson ? nullptr : buf[next], xprev, fprev, Xs + (long long)slot * n,
                 Fs + (long long)slot * n, 0.0, cj, omega, it > 0);
        if (!anderson) {
            cur = next;
            continue;
        }
        for (int j = 0; j < count; ++j) hslots[j] = ((head - count + j) % m + m) % m;
        std::memcpy(c->hscal + 512, hslots, sizeof(int) * 16);
        SDFT_CUDA(cudaMemcpyAsync(slots, c->hscal + 512, sizeof(int) * count, cudaMemcpyHostToDevice, c->stream));
        const int nblk = 64;
        anderson_gram_kernel<double><<<nblk, RB, 0, c->stream>>>(Fs, slots, count, r, cj, n, part);
        anderson_solve_kernel<<<1, 256, 0, c->stream>>>(part, nblk, count, gam, ffv);
        anderson_update_kernel<double><<<nblocks(n), 256, 0, c->stream>>>(buf[cur], r, cj, beta, Xs, Fs, slots, gam,
                                                                          count, n);
        SDFT_CUDA(cudaGetLastError());
        count_launch(c, 3);
        SDFT_CUDA(cudaMemcpyAsync(c->hscal, ffv, sizeof(double), cudaMemcpyDeviceToHost, c->stream));
        SDFT_CUDA(cudaEventRecord(read.e, c->stream));
        keep = cur;
        asked = it;
    }
    if (asked >= 0) {   // out of iterations with a residual unread
        const int at = asked;
        if (converged()) {
            cur = keep;
            it = at + 1;
        }
    }
    if (cur) SDFT_CUDA(cudaMemcpyAsync(phi, buf[cur], sizeof(double) * n, cudaMemcpyDeviceToDevice, c->stream));
    return it >= max_iter ? -it : it;
}

// ---------------------------------------------------------------------------------------
// Mixed-precision Poisson: FP64 residuals with FP32 AAR correction solves (iterative refinement).
//   r = rhs + L phi (FP64);  A delta = r solved approximately in FP32 by AAR;  phi += delta.
// Each refinement gains ~4-5 digits, so FP64-level residuals cost a few FP32 solves.
// ---------------------------------------------------------------------------------------
static int aar_fp32(sdft_ctx* c, const float* b, float* x, double tol_rel, int max_iter, double* final_rel) {
    const long long n = c->ng;
    const float omega = 0.6f, beta = 0.6f;
    const int m = 7, p = 6;
    float* r = c->work32 + 1 * n;
    float* xprev = c->work32 + 2 * n;
    float* fprev = c->work32 + 3 * n;
    float* Xs = c->work32 + 4 * n;
    float* Fs = Xs + (long long)m * n;
    double* gam = c->scal + 64;
    int* slots = (int*)(c->scal + 96);
    double* ffv = c->scal + 128;
    double* part = c->scal + 4096;
    const float cj = (float)(1.0 / (2.0 * c->coef.c0));
    double bnorm2;
    {
        // ||b||^2 through the history Gram with m = 0 (its last entry is (c f).(c f))
        anderson_gram_kernel<float><<<64, RB, 0, c->stream>>>(Fs, slots, 0, b, 1.0f, n, part);
        anderson_solve_kernel<<<1, 256, 0, c->stream>>>(part, 64, 0, gam, ffv);
        count_launch(c, 2);
        SDFT_CUDA(cudaMemcpyAsync(c->hscal, ffv, sizeof(double), cudaMemcpyDeviceToHost, c->stream));
        SDFT_CUDA(cudaStreamSynchronize(c->stream));
        bnorm2 = c->hscal[0];
    }
    SDFT_CUDA(cudaMemsetAsync(x, 0, sizeof(float) * n, c->stream));
    if (bnorm2 == 0.0) {
        *final_rel = 0.0;
        return 0;
    }
    int count = 0, head = 0, it = 0;
    int hslots[16];
    double rel = 1.0;
    for (it = 0; it < max_iter; ++it) {
        laplacian_residual<float>(c, x, b, r);
        const int slot = head;
        anderson_push_kernel<float><<<nblocks(n), 256, 0, c->stream>>>(x, r, cj, xprev, fprev, Xs + (long long)slot * n,
                                                                       Fs + (long long)slot * n, it > 0, n);
        count_launch(c);
        if (it > 0) {
            head = (head + 1) % m;
            count = std::min(count + 1, m);
        }
        const bool anderson = ((it + 1) % p == 0) && count > 0;
        if (anderson) {
            for (int j = 0; j < count; ++j) hslots[j] = ((head - count + j) % m + m) % m;
            std::memcpy(c->hscal + 512, hslots, sizeof(int) * 16);
            SDFT_CUDA(cudaMemcpyAsync(slots, c->hscal + 512, sizeof(int) * count, cudaMemcpyHostToDevice, c->stream));
            const int nblk = 64;
            anderson_gram_kernel<float><<<nblk, RB, 0, c->stream>>>(Fs, slots, count, r, cj, n, part);
            anderson_solve_kernel<<<1, 256, 0, c->stream>>>(part, nblk, count, gam, ffv);
            anderson_update_kernel<float><<<nblocks(n), 256, 0, c->stream>>>(x, r, cj, beta, Xs, Fs, slots, gam, count, n);
            SDFT_CUDA(cudaGetLastError());
            count_launch(c, 3);
            SDFT_CUDA(cudaMemcpyAsync(c->hscal, ffv, sizeof(double), cudaMemcpyDeviceToHost, c->stream));
            SDFT_CUDA(cudaStreamSynchronize(c->stream));
            rel = std::sqrt(c->hscal[0] / ((double)cj * cj) / bnorm2);
            if (!std::isfinite(rel)) throw Error{SDFT_ERR_NONFINITE, "Poisson residual is not finite"};
            if (rel <= tol_rel) {
                ++it;
                break;
            }
        } else {
            axpby_kernel<float><<<nblocks(n), 256, 0, c->stream>>>(x, r, omega * cj, 1.0f, n);
            SDFT_CUDA(cudaGetLastError());
            count_launch(c);
        }
    }
    *final_rel = rel;
    return it;
}

void laplacian_residual_f32(sdft_ctx* c, const float* x, const float* b, float* r) {
    laplacian_residual<float>(c, x, b, r);
}

// ---- FP64 passes of the refinement, each with the sum it needs (part[block][k], added by total_kernel) ----
template <int K>
__device__ __forceinline__ void block_total(const double (&v)[K], double* __restrict__ part) {
    __shared__ double sh[K][RB / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        double s = v[k];
        for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
        if (lane == 0) sh[k][warp] = s;
    }
    __syncthreads();
    if (threadIdx.x < K) {
        double s = 0.0;
        for (int w = 0; w < RB / 32; ++w) s += sh[threadIdx.x][w];
        part[(long long)blockIdx.x * K + threadIdx.x] = s;
    }
}
// out[k] = sum of part[block][k] over nblk blocks, K <= 2 quantities; one CTA of RB threads
__global__ void __launch_bounds__(RB) total_kernel(const double* __restrict__ part, int nblk, int K,
                                                   double* __restrict__ out) {
    double v[2] = {0.0, 0.0};
    for (int b = threadIdx.x; b < nblk; b += RB)
        for (int k = 0; k < K; ++k) v[k] += part[(long long)b * K + k];
    block_total<2>(v, out);   // two values at out[0], out[1]
}
// sums of a and b (b null: of a alone, K = 1 layout)
__global__ void __launch_bounds__(RB) sum2_kernel(const double* __restrict__ a, const double* __restrict__ b, long long n,
                                                  double* __restrict__ part) {
    double v[2] = {0.0, 0.0};
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        v[0] += a[i];
        if (b) v[1] += b[i];
    }
    if (b) block_total<2>(v, part);
    else block_total<1>({v[0]}, part);
}
// rhs = 4 pi (f - mean f), phi -= mean phi (sums = sum f, sum phi), and the sum of rhs^2
__global__ void __launch_bounds__(RB) poisson_rhs_kernel(const double* __restrict__ f, double* __restrict__ phi,
                                                         double* __restrict__ rhs, const double* __restrict__ sums,
                                                         long long n, double* __restrict__ part) {
    const double mf = sums[0] / (double)n, mp = sums[1] / (double)n;
    double v[1] = {0.0};
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const double r = 4.0 * M_PI * (f[i] - mf);
        rhs[i] = r;
        phi[i] -= mp;
        v[0] = fma(r, r, v[0]);
    }
    block_total<1>(v, part);
}
// r = rhs + L phi: its FP32 copy and the sum of r^2
__global__ void __launch_bounds__(RB) refine_residual_kernel(const double* __restrict__ phi,
                                                             const double* __restrict__ rhs, float* __restrict__ r32,
                                                             const __grid_constant__ LapCoef K, int n1, int n2, int n3,
                                                             double* __restrict__ part) {
    const int ng = n1 * n2 * n3;
    double v[1] = {0.0};
    for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < ng; g += gridDim.x * blockDim.x) {
        const double r = laplacian_residual_at<double, false>(phi, rhs, K, n1, n2, n3, 0.0, g);
        r32[g] = (float)r;
        v[0] = fma(r, r, v[0]);
    }
    block_total<1>(v, part);
}

// FP32 AAR with the multigrid preconditioner M (one V-cycle, poisson_mg.cu) in place of the Jacobi
// scaling: f_k = M r_k enters the Richardson steps x += omega f and the Anderson extrapolation every
// p-th step exactly where c r_k does in aar_fp32; convergence is tested on the true residual
// ||r_k|| / ||b|| at the Anderson steps.  With M A well conditioned a short history and frequent
// Anderson steps suffice.
static int aar_fp32_mg(sdft_ctx* c, const float* b, float* x, double tol_rel, int max_iter, double* final_rel) {
    const long long n = c->ng;
    const float omega = 0.7f, beta = 0.7f;
    const int m = 5, p = 3;
    // reduction grids: the history Gram's partials (m (m + 1) / 2 + m + 1 = 21 per block) fill NB * 21 of the
    // 12 288 doubles from scal + 4096, the residual's NB of the 1 024 from scal + 2048
    constexpr int NB = 152;
    float* r = c->work32 + 1 * n;
    float* xprev = c->work32 + 2 * n;
    float* fprev = c->work32 + 3 * n;
    float* Xs = c->work32 + 4 * n;
    float* Fs = Xs + (long long)m * n;
    float* z = c->work32 + 19 * n;
    double* gam = c->scal + 64;
    int* slots = (int*)(c->scal + 96);
    double* ffv = c->scal + 128;
    double* rrv = c->scal + 136;
    double* part = c->scal + 4096;
    double* part_r = c->scal + 2048;
    double bnorm2;
    {
        anderson_gram_kernel<float><<<NB, RB, 0, c->stream>>>(Fs, slots, 0, b, 1.0f, n, part_r);
        anderson_solve_kernel<<<1, 256, 0, c->stream>>>(part_r, NB, 0, gam, rrv);
        count_launch(c, 2);
        SDFT_CUDA(cudaMemcpyAsync(c->hscal, rrv, sizeof(double), cudaMemcpyDeviceToHost, c->stream));
        SDFT_CUDA(cudaStreamSynchronize(c->stream));
        bnorm2 = c->hscal[0];
    }
    SDFT_CUDA(cudaMemsetAsync(x, 0, sizeof(float) * n, c->stream));
    if (bnorm2 == 0.0) {
        *final_rel = 0.0;
        return 0;
    }
    int count = 0, head = 0, it = 0;
    int hslots[16];
    double rel = 1.0;
    for (it = 0; it < max_iter; ++it) {
        mg_residual_vcycle(c, x, b, r, z);
        const int slot = head;
        if (it > 0) {
            head = (head + 1) % m;
            count = std::min(count + 1, m);
        }
        const bool anderson = ((it + 1) % p == 0) && count > 0;
        mg_finish(c, r, z, x, xprev, fprev, Xs + (long long)slot * n, Fs + (long long)slot * n, omega, it > 0, !anderson);
        if (!anderson) continue;
        for (int j = 0; j < count; ++j) hslots[j] = ((head - count + j) % m + m) % m;
        std::memcpy(c->hscal + 512, hslots, sizeof(int) * 16);
        SDFT_CUDA(cudaMemcpyAsync(slots, c->hscal + 512, sizeof(int) * count, cudaMemcpyHostToDevice, c->stream));
        // the history Gram, and ||r||^2 of the residual this step was taken from
        anderson_gram2_kernel<float><<<dim3(NB, 2), RB, 0, c->stream>>>(Fs, slots, count, z, r, 1.0f, n, part, part_r);
        anderson_solve2_kernel<<<2, 256, 0, c->stream>>>(part, part_r, NB, count, gam, ffv, rrv);
        anderson_update_kernel<float><<<nblocks(n), 256, 0, c->stream>>>(x, z, 1.0f, beta, Xs, Fs, slots, gam, count, n);
        SDFT_CUDA(cudaGetLastError());
        count_launch(c, 3);
        SDFT_CUDA(cudaMemcpyAsync(c->hscal, rrv, sizeof(double), cudaMemcpyDeviceToHost, c->stream));
        SDFT_CUDA(cudaStreamSynchronize(c->stream));
        rel = std::sqrt(c->hscal[0] / bnorm2);
        if (!std::isfinite(rel)) throw Error{SDFT_ERR_NONFINITE, "Poisson residual is not finite"};
        if (rel <= tol_rel) {
            ++it;
            break;
        }
    }
    *final_rel = rel;
    return it;
}

// ---------------------------------------------------------------------------------------
// Persistent FP32 AAR: the whole correction solve A d = b (A = -L_h) in one cooperative launch.
// CTA k owns points [k*per, (k+1)*per).  Per iteration: residual r = b + L x_cur on own points
// (neighbours read from L2), history push, then Richardson x_next = x_cur + w c r or, every p-th
// iteration, Anderson x_next = x_cur + beta c r - sum gamma (X + beta F) with the small Gram
// reduced through per-block partials (every CTA sums them in the same order and solves the same
// m x m system).  x is double-buffered, so one grid barrier per iteration separates the reads of
// x_cur from the writes of x_next (two on Anderson steps).  The barrier spin is bounded: on
// timeout the kernel records an error status and every CTA returns.
// ---------------------------------------------------------------------------------------
struct AarPersistArgs {
    const float* b;
    float* x0;       // x buffers (double-buffered)
    float* x1;
    float* r;
    float* xprev;
    float* fprev;
    float* Xs;       // [m][n]
    float* Fs;       // [m][n]
    double* part;    // [gridDim][ND]
    unsigned* bar;   // [2]: arrival count, generation
    int* status;     // [4]: 0 ok / 1 barrier timeout, iterations, final buffer index
    double* rel_out;
    LapCoef K;
    int n1, n2, n3;
    long long n;
    float cj, omega, beta;
    double bnorm2, tol_rel;
    int max_iter;
    unsigned expected_blocks;   // arrivals the barrier waits for (== gridDim.x)
    long long spin_limit;
};

constexpr int AAR_M = 7, AAR_P = 6, AAR_ND = AAR_M * (AAR_M + 1) / 2 + AAR_M + 1;

__device__ bool grid_barrier(unsigned* bar, unsigned expected, long long limit, int* flag) {
    __shared__ int ok_s;
    __syncthreads();
    if (threadIdx.x == 0) {
        int ok = 1;
        volatile unsigned* gen = bar + 1;
        const unsigned g = *gen;
        __threadfence();
        const unsigned arrived = atomicAdd(bar, 1u);
        if (arrived == expected - 1) {
            atomicExch(bar, 0u);
            __threadfence();
            atomicAdd(bar + 1, 1u);
        } else {
            long long i = 0;
            while (*gen == g) {
                if (++i > limit || *(volatile int*)flag != 0) {
                    ok = 0;
                    break;
                }
            }
        }
        __threadfence();
        if (!ok) atomicExch(flag, 1);
        ok_s = ok;
    }
    __syncthreads();
    return ok_s != 0;
}

constexpr int AAR_BS = 256;    // threads per CTA of the persistent solver (one CTA per SM)

__global__ void __launch_bounds__(AAR_BS) aar_persistent_kernel(AarPersistArgs A) {
    __shared__ double red[AAR_ND][AAR_BS / 32];
    __shared__ double gam_s[AAR_M];
    __shared__ double ff_s;
    const long long per = (A.n + gridDim.x - 1) / gridDim.x;
    const long long lo = blockIdx.x * per, hi = min(A.n, lo + per);
    int head = 0, count = 0;
    int cur = 0;
    int it;
    double rel = 1.0;
    for (it = 0; it < A.max_iter; ++it) {
        float* xc = cur ? A.x1 : A.x0;
        float* xn = cur ? A.x0 : A.x1;
        const int slot = head;
        // residual and history push on own points.  Grid coordinates advance incrementally in
        // 32-bit arithmetic (the points of a thread are blockDim apart), so no division per point.
        {
            const int n1 = A.n1, n2 = A.n2, n3 = A.n3;
            const int pl32 = n1 * n2;
            int g = (int)lo + (int)threadIdx.x;
            int i = g % n1, row = g / n1;
            int j = row % n2, k = row / n2;
            const int di = (int)(blockDim.x % (unsigned)n1), drow = (int)(blockDim.x / (unsigned)n1);
            const int dj = drow % n2, dk = drow / n2;
            for (; g < (int)hi; g += (int)blockDim.x) {
                const int rowbase = g - i;              // (k n2 + j) n1
                const int colbase = g - j * n1;         // k n1 n2 + i
                const int plbase = g - k * pl32;        // j n1 + i
                float acc = (float)A.K.c0 * xc[g];
#pragma unroll
                for (int rr = 1; rr <= FD_RADIUS; ++rr) {
                    int ip = i + rr, im = i - rr, jp = j + rr, jm = j - rr, kp = k + rr, km = k - rr;
                    ip -= ip >= n1 ? n1 : 0;
                    im += im < 0 ? n1 : 0;
                    jp -= jp >= n2 ? n2 : 0;
                    jm += jm < 0 ? n2 : 0;
                    kp -= kp >= n3 ? n3 : 0;
                    km += km < 0 ? n3 : 0;
                    acc += (float)A.K.c[0][rr] * (xc[rowbase + ip] + xc[rowbase + im]);
                    acc += (float)A.K.c[1][rr] * (xc[colbase + jp * n1] + xc[colbase + jm * n1]);
                    acc += (float)A.K.c[2][rr] * (xc[plbase + kp * pl32] + xc[plbase + km * pl32]);
                }
                const float r = A.b[g] - 2.f * acc;
                A.r[g] = r;
                const float fi = A.cj * r;
                if (it > 0) {
                    A.Xs[(long long)slot * A.n + g] = xc[g] - A.xprev[g];
                    A.Fs[(long long)slot * A.n + g] = fi - A.fprev[g];
                }
                A.xprev[g] = xc[g];
                A.fprev[g] = fi;
                // next point of this thread: blockDim further along x, then y, then z
                i += di;
                j += dj;
                k += dk;
                if (i >= n1) {
                    i -= n1;
                    ++j;
                }
                if (j >= n2) {
                    j -= n2;
                    ++k;
                }
            }
        }
        if (it > 0) {
            head = (head + 1) % AAR_M;
            count = min(count + 1, AAR_M);
        }
        const bool anderson = ((it + 1) % AAR_P == 0) && count > 0;
        if (!anderson) {
            for (long long g = lo + threadIdx.x; g < hi; g += blockDim.x) xn[g] = xc[g] + A.omega * A.cj * A.r[g];
        } else {
            // partial Gram of the history (slots in age order) and F.(c r), (c r).(c r)
            int sl[AAR_M];
            for (int jj = 0; jj < count; ++jj) sl[jj] = ((head - count + jj) % AAR_M + AAR_M) % AAR_M;
            const int nd = count * (count + 1) / 2 + count + 1;
            double* row = A.part + (long long)blockIdx.x * nd;
            switch (count) {
#define SDFT_AAR_CASE(CC) \
    case CC: gram_accum<CC, AAR_BS / 32>(A.Fs, sl, A.r, A.cj, A.n, lo + threadIdx.x, hi, blockDim.x, row, red); break;
                SDFT_AAR_CASE(1) SDFT_AAR_CASE(2) SDFT_AAR_CASE(3) SDFT_AAR_CASE(4) SDFT_AAR_CASE(5) SDFT_AAR_CASE(6)
                SDFT_AAR_CASE(7)
#undef SDFT_AAR_CASE
                default: break;
            }
            if (!grid_barrier(A.bar, A.expected_blocks, A.spin_limit, A.status)) return;
            anderson_solve_block(A.part, gridDim.x, count, gam_s, &ff_s);
            __syncthreads();
            rel = sqrt(ff_s / ((double)A.cj * A.cj) / A.bnorm2);
            for (long long g = lo + threadIdx.x; g < hi; g += blockDim.x) {
                float v = xc[g] + A.beta * A.cj * A.r[g];
                for (int jj = 0; jj < count; ++jj) {
                    const long long o = (long long)sl[jj] * A.n + g;
                    v -= (float)gam_s[jj] * (A.Xs[o] + A.beta * A.Fs[o]);
                }
                xn[g] = v;
            }
        }
        if (!grid_barrier(A.bar, A.expected_blocks, A.spin_limit, A.status)) return;
        cur ^= 1;
        if (anderson && !(rel > A.tol_rel)) {   // converged (also stops on NaN)
            ++it;
            break;
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        A.status[1] = it;
        A.status[2] = cur;
        *A.rel_out = rel;
    }
}

// FP32 correction solve by the persistent kernel; x (work32 slot) receives the solution.
static int aar_fp32_persistent(sdft_ctx* c, const float* b, float* x, double tol_rel, int max_iter,
                               double* final_rel) {
    const long long n = c->ng;
    AarPersistArgs A;
    A.b = b;
    A.x0 = x;
    A.x1 = c->work32 + 19 * n;
    A.r = c->work32 + 1 * n;
    A.xprev = c->work32 + 2 * n;
    A.fprev = c->work32 + 3 * n;
    A.Xs = c->work32 + 4 * n;
    A.Fs = A.Xs + (long long)AAR_M * n;
    A.part = c->scal + 4096;
    A.bar = reinterpret_cast<unsigned*>(c->scal + 40);
    A.status = reinterpret_cast<int*>(c->scal + 42);
    A.rel_out = c->scal + 44;
    A.K = lap_coef<double>(c);
    A.n1 = c->n[0];
    A.n2 = c->n[1];
    A.n3 = c->n[2];
    A.n = n;
    A.cj = (float)(1.0 / (2.0 * c->coef.c0));
    A.omega = 0.6f;
    A.beta = 0.6f;
    A.tol_rel = tol_rel;
    A.max_iter = max_iter;
    A.spin_limit = 1LL << 24;   // volatile polls of the barrier generation (~0.1-1 s)
    // ||b||^2
    {
        double* part = c->scal + 2048;
        anderson_gram_kernel<float><<<64, RB, 0, c->stream>>>(A.Fs, nullptr, 0, b, 1.0f, n, part);
        anderson_solve_kernel<<<1, 256, 0, c->stream>>>(part, 64, 0, c->scal + 64, c->scal + 128);
        count_launch(c, 2);
        SDFT_CUDA(cudaMemcpyAsync(c->hscal, c->scal + 128, sizeof(double), cudaMemcpyDeviceToHost, c->stream));
        SDFT_CUDA(cudaStreamSynchronize(c->stream));
        A.bnorm2 = c->hscal[0];
    }
    SDFT_CUDA(cudaMemsetAsync(x, 0, sizeof(float) * n, c->stream));
    if (A.bnorm2 == 0.0) {
        *final_rel = 0.0;
        return 0;
    }
    // grid: co-resident CTAs (cooperative launch), at most one per 2048 points, <= 12288 partial slots
    int dev = 0, nsm = 0, per_sm = 0;
    SDFT_CUDA(cudaGetDevice(&dev));
    SDFT_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    SDFT_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, aar_persistent_kernel, AAR_BS, 0));
    if (per_sm < 1) {
        c->aar_persistent = false;
        return aar_fp32(c, b, x, tol_rel, max_iter, final_rel);
    }
    // every co-resident CTA (latency hiding for the stencil's scattered loads), fewer for small grids
    SDFT_REQUIRE(n < (1LL << 31) - 4096, SDFT_ERR_INVALID_ARG, "persistent Poisson solver: grid too large");
    long long nblk = std::min<long long>((long long)nsm * per_sm, (n + 1023) / 1024);
    nblk = std::max<long long>(1, std::min<long long>(nblk, 12288 / AAR_ND));
    A.expected_blocks = (unsigned)nblk + (c->test_barrier_extra ? 1u : 0u);
    if (c->test_barrier_extra) A.spin_limit = 200000;
    SDFT_CUDA(cudaMemsetAsync(A.bar, 0, 2 * sizeof(unsigned), c->stream));
    SDFT_CUDA(cudaMemsetAsync(A.status, 0, 4 * sizeof(int), c->stream));
    void* args[] = {&A};
    const cudaError_t le = cudaLaunchCooperativeKernel((const void*)aar_persistent_kernel, dim3((unsigned)nblk),
                                                       dim3(AAR_BS), args, 0, c->stream);
    if (le != cudaSuccess) {
        // no co-residency guarantee available: fall back to one launch per iteration
        cudaGetLastError();
        c->aar_persistent = false;
        return aar_fp32(c, b, x, tol_rel, max_iter, final_rel);
    }
    count_launch(c);
    int st[4];
    SDFT_CUDA(cudaMemcpyAsync(st, A.status, sizeof(st), cudaMemcpyDeviceToHost, c->stream));
    SDFT_CUDA(cudaMemcpyAsync(c->hscal, A.rel_out, sizeof(double), cudaMemcpyDeviceToHost, c->stream));
    SDFT_CUDA(cudaStreamSynchronize(c->stream));
    if (st[0] != 0) throw Error{SDFT_ERR_DEVICE_TIMEOUT, "persistent Poisson solver: grid barrier timed out"};
    if (st[2] == 1) SDFT_CUDA(cudaMemcpyAsync(x, A.x1, sizeof(float) * n, cudaMemcpyDeviceToDevice, c->stream));
    *final_rel = c->hscal[0];
    return st[1];
}

int poisson_mixed(sdft_ctx* c, const double* f, double* phi, double tol, int max_iter) {
    const long long n = c->ng;
    ScopedTimer timer(c, SDFT_K_POISSON);
    double* rhs = c->work64 + 0 * n;
    float* b32 = c->work32;
    float* d32 = c->work32 + 18 * n;
    double* part = c->scal + 2048;    // partial sums of two quantities, PB blocks
    double* sums = c->scal + 1536;
    constexpr int PB = 256;
    auto host_sums = [&](int k) {
        SDFT_CUDA(cudaGetLastError());
        SDFT_CUDA(cudaMemcpyAsync(c->hscal, sums, sizeof(double) * k, cudaMemcpyDeviceToHost, c->stream));
        SDFT_CUDA(cudaStreamSynchronize(c->stream));
    };
    // sums[0, 1] = sum f, sum phi;  rhs = 4 pi (f - mean f), phi -= mean(phi), with the sum of rhs^2
    sum2_kernel<<<PB, RB, 0, c->stream>>>(f, phi, n, part);
    total_kernel<<<1, 256, 0, c->stream>>>(part, PB, 2, sums);
    poisson_rhs_kernel<<<PB, RB, 0, c->stream>>>(f, phi, rhs, sums, n, part);
    total_kernel<<<1, 256, 0, c->stream>>>(part, PB, 1, sums);
    count_launch(c, 4);
    host_sums(1);
    const double bnorm2 = c->hscal[0];
    if (bnorm2 == 0.0) {
        SDFT_CUDA(cudaMemsetAsync(phi, 0, sizeof(double) * n, c->stream));
        return 0;
    }
    // zero-mean gauge: FP32 corrections drift along the constant null vector of L, which the
    // residual cannot see, so the mean is removed from phi at the end
    auto remove_mean = [&]() {
        sum2_kernel<<<PB, RB, 0, c->stream>>>(phi, nullptr, n, part);
        total_kernel<<<1, 256, 0, c->stream>>>(part, PB, 1, sums);
        add_scalar_kernel<<<nblocks(n), 256, 0, c->stream>>>(phi, sums, -1.0 / (double)n, n);
        SDFT_CUDA(cudaGetLastError());
        count_launch(c, 3);
    };
    const LapCoef K = lap_coef<double>(c);
    int total = 0;
    for (int refine = 0; refine < 16; ++refine) {
        // FP64 residual r = rhs + L phi: its norm, and its FP32 copy as the next correction's right-hand side
        refine_residual_kernel<<<(unsigned)std::min<long long>((n + RB - 1) / RB, 1024), RB, 0, c->stream>>>(
            phi, rhs, b32, K, c->n[0], c->n[1], c->n[2], part);
        total_kernel<<<1, 256, 0, c->stream>>>(part, (int)std::min<long long>((n + RB - 1) / RB, 1024), 1, sums);
        count_launch(c, 2);
        host_sums(1);
        const double rel = std::sqrt(c->hscal[0] / bnorm2);
        if (!std::isfinite(rel)) throw Error{SDFT_ERR_NONFINITE, "Poisson residual is not finite"};
        if (rel <= tol) {
            remove_mean();
            return std::max(total, 1);
        }
        if (total >= max_iter) break;
        // FP32 correction A d = r: a relative reduction of 1e-3 per refinement stays above the
        // FP32 rounding floor of the residual (~ cond(L) * 2^-24)
        double inner_rel = 1.0;
        const double want = std::max(1e-3, 0.3 * tol / rel);
        const int budget = std::min(400, max_iter - total);
        total += !c->mg.empty()       ? aar_fp32_mg(c, b32, d32, want, budget, &inner_rel)
                 : c->aar_persistent ? aar_fp32_persistent(c, b32, d32, want, budget, &inner_rel)
                                     : aar_fp32(c, b32, d32, want, budget, &inner_rel);
        convert_add_kernel<double, float><<<nblocks(n), 256, 0, c->stream>>>(phi, d32, 1.0, 1.0, n);
        count_launch(c);
    }
    remove_mean();
    return -std::max(total, 1);
}

void density_accumulate(sdft_ctx* c, int precision, bool cplx, const void* X, const double* occ, int ncol,
                        double weight, double* rho) {
    const double scale = weight / c->dV;
    const unsigned nb = nblocks(c->ng);
    ScopedTimer timer(c, SDFT_K_DENSITY, (double)block_elems_bytes(c, precision, cplx, ncol));
    const size_t sm32 = sizeof(float) * (size_t)ncol;   // FP32 copy of the occupations
    SDFT_REQUIRE(sm32 <= 48 * 1024, SDFT_ERR_INVALID_ARG, "density: too many states for one block's occupations");
    if (precision == SDFT_FP64) {
        if (cplx) density_kernel<1><<<nb, 256, 0, c->stream>>>(X, occ, ncol, scale, c->ng, rho);
        else density_kernel<0><<<nb, 256, 0, c->stream>>>(X, occ, ncol, scale, c->ng, rho);
    } else {
        if (cplx) density_kernel<3><<<nb, 256, sm32, c->stream>>>(X, occ, ncol, scale, c->ng, rho);
        else density_kernel<2><<<nb, 256, sm32, c->stream>>>(X, occ, ncol, scale, c->ng, rho);
    }
    SDFT_CUDA(cudaGetLastError());
    count_launch(c);
}

void fermi_device(sdft_ctx* c, const double* eig, double* occ, double* out) {
    const int nk = c->opt.nkpt;
    double* kw = c->scal + 256;
    SDFT_CUDA(cudaMemcpyAsync(kw, c->kw.data(), sizeof(double) * nk, cudaMemcpyHostToDevice, c->stream));
    const double fs = c->opt.nspin == 1 ? 2.0 : 1.0;
    fermi_kernel<<<1, 256, 0, c->stream>>>(eig, kw, c->opt.nspin, nk, c->opt.nstates, c->nelec, c->opt.kT, fs, occ,
                                           out);
    SDFT_CUDA(cudaGetLastError());
    count_launch(c);
}

// ---------------------------------------------------------------------------------------
// Kerker preconditioner of the mixing (paper Sec. 2.1: periodic Pulay with a real-space
// preconditioner of Kerker type): P f = (-L_h)(-L_h + k0^2)^-1 f = f - k0^2 y, (-L_h + k0^2) y = f.
// The screened operator is positive definite, so y comes from the same AAR iteration as the
// Poisson solve (Jacobi-preconditioned Richardson steps, Anderson extrapolation every p-th step),
// with the diagonal shift k0^2 in the residual and in the Jacobi factor; no gauge is involved.
// ---------------------------------------------------------------------------------------
namespace {
constexpr int KERKER_M = 7, KERKER_P = 6;
constexpr double KERKER_TOL = 1e-10;    // relative residual of the screened solve inside the SCF

// x_k ← x_k - sum_j gamma_j X_j and f ← beta (f - sum_j gamma_j F_j): the optimal residual form of a
// Pulay step, whose linear part is then preconditioned
__global__ void pulay_residual_kernel(double* __restrict__ x, double* __restrict__ f, const double* __restrict__ X,
                                      const double* __restrict__ F, const int* __restrict__ slots,
                                      const double* __restrict__ gamma, int m, double beta, long long n) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        double xv = x[i], fv = f[i];
        for (int j = 0; j < m; ++j) {
            const long long o = (long long)slots[j] * n + i;
            xv -= gamma[j] * X[o];
            fv -= gamma[j] * F[o];
        }
        x[i] = xv;
        f[i] = beta * fv;
    }
}
}  // namespace

static double* kerker_workspace(sdft_ctx* c) {
    // rhs copy, solution, AAR residual, previous iterate and residual, X[m], F[m]
    if (!c->kerker_ws) c->kerker_ws = (double*)ctx_alloc(c, sizeof(double) * (size_t)(5 + 2 * KERKER_M) * c->ng);
    return c->kerker_ws;
}

int kerker_apply(sdft_ctx* c, const double* f, double* out, double k0, double tol, int max_iter) {
    const long long n = c->ng;
    SDFT_REQUIRE(k0 > 0.0 && tol > 0.0 && max_iter >= 1, SDFT_ERR_INVALID_ARG, "Kerker: k0 > 0, tol > 0 required");
    double* ws = kerker_workspace(c);
    double* y = ws + 1 * n;
    double* r = ws + 2 * n;
    double* xprev = ws + 3 * n;
    double* fprev = ws + 4 * n;
    double* Xs = ws + 5 * n;
    double* Fs = Xs + (long long)KERKER_M * n;
    double* gam = c->scal + 64;
    int* slots = (int*)(c->scal + 96);
    double* ffv = c->scal + 128;
    double* part = c->scal + 4096;
    const double k2 = k0 * k0;
    const double cj = 1.0 / (2.0 * c->coef.c0 + k2);   // Jacobi: diag(-L_h + k0^2)
    const double omega = 0.6, beta = 0.6;
    double bnorm2;
    {
        const double* A[1] = {f};
        dots_host(c, 1, A, A, n, &bnorm2);
    }
    SDFT_CUDA(cudaMemsetAsync(y, 0, sizeof(double) * n, c->stream));
    int it = 0;
    if (bnorm2 > 0.0) {
        int count = 0, head = 0;
        int hslots[16];
        bool done = false;
        for (it = 0; it < max_iter; ++it) {
            laplacian_residual<double>(c, y, f, r, k2);
            anderson_push_kernel<double><<<nblocks(n), 256, 0, c->stream>>>(y, r, cj, xprev, fprev,
                                                                            Xs + (long long)head * n,
                                                                            Fs + (long long)head * n, it > 0, n);
            count_launch(c);
            if (it > 0) {
                head = (head + 1) % KERKER_M;
                count = std::min(count + 1, KERKER_M);
            }
            if (((it + 1) % KERKER_P == 0) && count > 0) {
                for (int j = 0; j < count; ++j) hslots[j] = ((head - count + j) % KERKER_M + KERKER_M) % KERKER_M;
                std::memcpy(c->hscal + 512, hslots, sizeof(int) * 16);
                SDFT_CUDA(cudaMemcpyAsync(slots, c->hscal + 512, sizeof(int) * count, cudaMemcpyHostToDevice, c->stream));
                anderson_gram_kernel<double><<<64, RB, 0, c->stream>>>(Fs, slots, count, r, cj, n, part);
                anderson_solve_kernel<<<1, 256, 0, c->stream>>>(part, 64, count, gam, ffv);
                anderson_update_kernel<double><<<nblocks(n), 256, 0, c->stream>>>(y, r, cj, beta, Xs, Fs, slots, gam,
                                                                                  count, n);
                SDFT_CUDA(cudaGetLastError());
                count_launch(c, 3);
                SDFT_CUDA(cudaMemcpyAsync(c->hscal, ffv, sizeof(double), cudaMemcpyDeviceToHost, c->stream));
                SDFT_CUDA(cudaStreamSynchronize(c->stream));
                const double rn2 = c->hscal[0] / (cj * cj);
                if (!std::isfinite(rn2)) throw Error{SDFT_ERR_NONFINITE, "Kerker solve residual is not finite"};
                if (rn2 <= tol * tol * bnorm2) {
                    ++it;
                    done = true;
                    break;
                }
            } else {
                axpby_kernel<double><<<nblocks(n), 256, 0, c->stream>>>(y, r, omega * cj, 1.0, n);
                SDFT_CUDA(cudaGetLastError());
                count_launch(c);
            }
        }
        if (!done) return -it;
    }
    // out = f - k0^2 y
    SDFT_CUDA(cudaMemcpyAsync(out, f, sizeof(double) * n, cudaMemcpyDeviceToDevice, c->stream));
    axpby_kernel<double><<<nblocks(n), 256, 0, c->stream>>>(out, y, -k2, 1.0, n);
    SDFT_CUDA(cudaGetLastError());
    count_launch(c);
    return std::max(it, 1);
}

// Pulay mixing on rho_in (paper Sec. 2.1; Banerjee et al. 2016, Pratapa & Suryanarayana 2015):
// f = rho_out - rho_in; linear step rho += beta f, or Pulay every period-th iteration.
void pulay_update(sdft_ctx* c) {
    const long long n = (long long)c->opt.nspin * c->ng;
    const int m = c->opt.mix_hist;
    double* f = c->work64;  // needs nspin*ng <= 2 ng: use work64[0 .. 2ng)
    // f = rho_out - rho_in
    SDFT_CUDA(cudaMemcpyAsync(f, c->rho_out, sizeof(double) * n, cudaMemcpyDeviceToDevice, c->stream));
    axpby_kernel<double><<<nblocks(n), 256, 0, c->stream>>>(f, c->rho_in, -1.0, 1.0, n);
    count_launch(c);
    const int slot = c->mix_head;
    anderson_push_kernel<double><<<nblocks(n), 256, 0, c->stream>>>(c->rho_in, f, 1.0, c->mix_xprev, c->mix_fprev,
                                                            c->mix_dx + (long long)slot * n,
                                                            c->mix_df + (long long)slot * n, c->mix_k > 0, n);
    count_launch(c);
    if (c->mix_k > 0) {
        c->mix_head = (c->mix_head + 1) % m;
        c->mix_count = std::min(c->mix_count + 1, m);
    }
    const bool pulay = c->mix_k > 0 && c->mix_count > 0 && ((c->mix_k + 1) % c->opt.pulay_period == 0);
    if (c->opt.kerker_k0 > 0.0) {
        // Kerker-preconditioned form: x <- x - X gamma + P(beta (f - F gamma)), P channel by channel
        if (pulay) {
            int hslots[16];
            const int cnt = c->mix_count;
            for (int j = 0; j < cnt; ++j) hslots[j] = ((c->mix_head - cnt + j) % m + m) % m;
            int* slots = (int*)(c->scal + 160);
            double* gam = c->scal + 192;
            double* ffv = c->scal + 224;
            double* part = c->scal + 4096;
            std::memcpy(c->hscal + 640, hslots, sizeof(int) * 16);
            SDFT_CUDA(cudaMemcpyAsync(slots, c->hscal + 640, sizeof(int) * cnt, cudaMemcpyHostToDevice, c->stream));
            const int nblk = 32;
            anderson_gram_kernel<double><<<nblk, RB, 0, c->stream>>>(c->mix_df, slots, cnt, f, 1.0, n, part);
            anderson_solve_kernel<<<1, 256, 0, c->stream>>>(part, nblk, cnt, gam, ffv);
            pulay_residual_kernel<<<nblocks(n), 256, 0, c->stream>>>(c->rho_in, f, c->mix_dx, c->mix_df, slots, gam, cnt,
                                                                     c->opt.mix_beta, n);
            count_launch(c, 3);
            if (c->opt.pulay_restart) c->mix_count = 0;
        } else {
            axpby_kernel<double><<<nblocks(n), 256, 0, c->stream>>>(f, f, 0.0, c->opt.mix_beta, n);
            count_launch(c);
        }
        SDFT_CUDA(cudaGetLastError());
        double* pf = c->work64 + 2 * c->ng;   // P of one channel
        for (int sp = 0; sp < c->opt.nspin; ++sp) {
            const int it = kerker_apply(c, f + (long long)sp * c->ng, pf, c->opt.kerker_k0, KERKER_TOL, 4000);
            if (it < 0) throw Error{SDFT_ERR_NOT_CONVERGED, "Kerker screened-Poisson solve did not converge"};
            axpby_kernel<double><<<nblocks(c->ng), 256, 0, c->stream>>>(c->rho_in + (long long)sp * c->ng, pf, 1.0, 1.0,
                                                                        c->ng);
            count_launch(c);
        }
        SDFT_CUDA(cudaGetLastError());
        c->mix_k += 1;
        return;
    }
    if (pulay) {
        int hslots[16];
        const int cnt = c->mix_count;
        for (int j = 0; j < cnt; ++j) hslots[j] = ((c->mix_head - cnt + j) % m + m) % m;
        int* slots = (int*)(c->scal + 160);
        double* gam = c->scal + 192;
        double* ffv = c->scal + 224;
        double* part = c->scal + 4096;
        std::memcpy(c->hscal + 640, hslots, sizeof(int) * 16);
        SDFT_CUDA(cudaMemcpyAsync(slots, c->hscal + 640, sizeof(int) * cnt, cudaMemcpyHostToDevice, c->stream));
        const int nblk = 32;  // 32 x (m(m+1)/2 + m + 1) <= 12288 partials for m <= 16
        anderson_gram_kernel<double><<<nblk, RB, 0, c->stream>>>(c->mix_df, slots, cnt, f, 1.0, n, part);
        anderson_solve_kernel<<<1, 256, 0, c->stream>>>(part, nblk, cnt, gam, ffv);
        anderson_update_kernel<double><<<nblocks(n), 256, 0, c->stream>>>(c->rho_in, f, 1.0, c->opt.mix_beta, c->mix_dx,
                                                                  c->mix_df, slots, gam, cnt, n);
        count_launch(c, 3);
        if (c->opt.pulay_restart) {
            c->mix_count = 0;
        }
    } else {
        axpby_kernel<double><<<nblocks(n), 256, 0, c->stream>>>(c->rho_in, f, c->opt.mix_beta, 1.0, n);
        count_launch(c);
    }
    SDFT_CUDA(cudaGetLastError());
    c->mix_k += 1;
}

void forces_compute(sdft_ctx* c) {
    const int na = c->natom;
    c->forces.assign(3 * na, 0.0);
    double* dF = c->scal + 3072;  // up to 341 atoms
    SDFT_REQUIRE(3 * na <= 1024, SDFT_ERR_INVALID_ARG, "forces: too many atoms for the scalar area");
    for (int i = 0; i < 3 * na; ++i) c->hscal[i] = -c->dEsc[i];
    SDFT_CUDA(cudaMemcpyAsync(dF, c->hscal, sizeof(double) * 3 * na, cudaMemcpyHostToDevice, c->stream));
    std::vector<AtomG> at = atom_g(c);
    AtomG* dat = (AtomG*)ctx_alloc(c, sizeof(AtomG) * std::max(1, na));
    SDFT_CUDA(cudaMemcpyAsync(dat, at.data(), sizeof(AtomG) * na, cudaMemcpyHostToDevice, c->stream));
    // partial sums in the Gram's split-K buffer (free here): at most natom * ncol chunks of 3, and part holds
    // at least 128 ncol^2 and 2^20 doubles
    const int nloc = std::max(1, std::min(32, (4 * 152 + na - 1) / na));
    SDFT_REQUIRE((size_t)3 * na * std::max(nloc, c->opt.nstates) <= c->part_elems, SDFT_ERR_INVALID_ARG,
                 "forces: partial buffer too small");
    force_local_kernel<<<dim3(na, nloc), RB, 0, c->stream>>>(dat, c->n[0], c->n[1], c->n[2], c->h[0], c->h[1], c->h[2],
                                                             c->phi, c->part, c->opt.boundary == SDFT_BC_DIRICHLET);
    force_finish_kernel<<<na, 96, 0, c->stream>>>(c->part, nloc, c->dV, nullptr, dF);
    count_launch(c, 2);
    std::vector<double> rp2(na);
    for (int a = 0; a < na; ++a) rp2[a] = std::pow(c->species[c->types[a]].r_proj, 2);
    double* d_rp2 = (double*)ctx_alloc(c, sizeof(double) * std::max(1, na));
    double* d_pos = (double*)ctx_alloc(c, sizeof(double) * 3 * std::max(1, na));
    SDFT_CUDA(cudaMemcpyAsync(d_rp2, rp2.data(), sizeof(double) * na, cudaMemcpyHostToDevice, c->stream));
    SDFT_CUDA(cudaMemcpyAsync(d_pos, c->pos.data(), sizeof(double) * 3 * na, cudaMemcpyHostToDevice, c->stream));
    for (const Problem& P : c->probs) {
        const KBTables& T = c->kb[P.kpt];
        const void* X = c->opt.precision == SDFT_FP64 ? P.X : P.X64;
        SDFT_REQUIRE(X != nullptr, SDFT_ERR_INVALID_ARG, "forces need FP64 orbitals");
        const double wk = c->kw[P.kpt];
        // four real (two complex) columns per CTA; fewer when the cell is so small that the atoms times the
        // column groups would leave SMs idle
        const int ns = c->opt.nstates;
        auto launch = [&](auto kfn, int nc) {
            const int nchunk = (ns + nc - 1) / nc;
            kfn<<<dim3(na, nchunk), RB, 0, c->stream>>>(T.cnt, T.idx, T.img, T.val64, T.cap, (const double*)X, ns,
                                                        c->ng, P.occ, d_pos, d_rp2, c->n[0], c->n[1], c->n[2], c->h[0],
                                                        c->h[1], c->h[2], c->part);
            force_finish_kernel<<<na, 96, 0, c->stream>>>(c->part, nchunk, wk, T.gamma, dF);
        };
        const bool few = (long long)na * ns < 4 * 152;
        if (T.cplx && few) launch(force_nl_kernel<true, 1>, 1);
        else if (T.cplx) launch(force_nl_kernel<true, 2>, 2);
        else if (few) launch(force_nl_kernel<false, 1>, 1);
        else launch(force_nl_kernel<false, 4>, 4);
        count_launch(c, 2);
    }
    SDFT_CUDA(cudaGetLastError());
    SDFT_CUDA(cudaMemcpyAsync(c->hscal, dF, sizeof(double) * 3 * na, cudaMemcpyDeviceToHost, c->stream));
    SDFT_CUDA(cudaStreamSynchronize(c->stream));
    for (int i = 0; i < 3 * na; ++i) c->forces[i] = c->hscal[i];
    ctx_release(c, dat);   // per-call tables: released so that repeated SCFs (MD steps) do not accumulate them
    ctx_release(c, d_rp2);
    ctx_release(c, d_pos);
}

}  // namespace sdft
