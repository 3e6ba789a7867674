// Geometric multigrid V-cycle for the periodic Poisson problem: the preconditioner M ~ A^-1 of the
// FP32 AAR correction solves, A = -L_h the order-12 finite-difference Laplacian (paper Sec. 2.1:
// the electrostatic potential from a Poisson problem solved by AAR with matrix-free stencil
// Laplacian-vector products; the paper does not fix AAR's preconditioner, the plain choice being
// the Jacobi scaling 1 / diag A).
//
// M applies one V-cycle of the second-order (7-point) Laplacian A2 on a hierarchy of grids that
// halves every dimension while it is even: red-black Gauss-Seidel smoothing, full-weighting
// restriction of the residual, trilinear prolongation, and on the coarsest grid (at most 512
// points, or up to 16 384 when a dimension turns odd earlier) a fixed number of Chebyshev
// iterations for the known spectrum of A2, run by one CTA out of shared memory.  A2 and A share their low-frequency spectrum; at the highest grid frequency the
// order-12 symbol is about 2.5 times the second-order one, so the preconditioned operator M A
// keeps its eigenvalues in a small interval and AAR reaches a 1e-3 reduction in a few iterations
// instead of the hundreds the Jacobi scaling needs (its iteration count grows with the grid).
//
// Every grid is periodic, so A2 is singular with the constants as null space.  The right-hand
// sides the V-cycle sees have zero mean (residuals of a zero-mean problem; full weighting keeps
// the mean), and no smoothing or Chebyshev step adds a constant, so no projection is needed.
#include "internal.cuh"

#include <algorithm>
#include <cmath>
#include <cstdlib>

namespace sdft {
namespace {

struct MgDims {
    int n1, n2, n3;
    float w1, w2, w3;   // 1 / h_d^2 of the level
    float diag;         // 2 (w1 + w2 + w3)
};

__device__ __forceinline__ int wrapi(int i, int n) { return i < 0 ? i + n : (i >= n ? i - n : i); }

// (A2 x)[i, j, k] on a periodic grid
__device__ __forceinline__ float apply_a2(const float* __restrict__ x, const MgDims& d, int i, int j, int k) {
    const int rowj = (k * d.n2 + j) * d.n1;
    const float xc = x[rowj + i];
    const float sx = x[rowj + wrapi(i + 1, d.n1)] + x[rowj + wrapi(i - 1, d.n1)];
    const float sy = x[(k * d.n2 + wrapi(j + 1, d.n2)) * d.n1 + i] + x[(k * d.n2 + wrapi(j - 1, d.n2)) * d.n1 + i];
    const float sz = x[(wrapi(k + 1, d.n3) * d.n2 + j) * d.n1 + i] + x[(wrapi(k - 1, d.n3) * d.n2 + j) * d.n1 + i];
    return d.diag * xc - (d.w1 * sx + d.w2 * sy + d.w3 * sz);
}

// One red-black sweep before and one after the coarse correction, fused so that a level takes four launches of
// which each reads what it needs once (the plain form was seven: two half sweeps, restriction of the residual at
// every point, prolongation, two half sweeps; 20 to 25 launches and 74 us a cycle at 80^3, 53 us now):
//   * the sweep before starts from zero, so a red point is b / diag and a black one needs b alone: one pass;
//   * after it the residual of a black point is zero but for rounding, so the restriction visits the 13 red points
//     of the 27 of a coarse point's stencil (2I, 2J, 2K is red);
//   * in the sweep after (black, then red) a black point's new value needs the prolonged red neighbours and a red
//     point's the new black ones: the prolonged values are formed where they are read and never stored.
// Red points are those with even i + j + k; the levels that are swept have even dimensions, so a point's six
// neighbours have the other colour.
struct Pt {
    int i, j, k;
};
__device__ __forceinline__ Pt point_of(int t, int n1, int n2) {
    const int row = t / n1;
    Pt p;
    p.i = t - row * n1;
    p.k = row / n2;
    p.j = row - p.k * n2;
    return p;
}
// the six neighbours' values f(i, j, k), weighted by the level's 1 / h^2
template <typename F>
__device__ __forceinline__ float neighbours(const MgDims& d, Pt p, F f) {
    float s = d.w1 * (f(wrapi(p.i + 1, d.n1), p.j, p.k) + f(wrapi(p.i - 1, d.n1), p.j, p.k));
    s += d.w2 * (f(p.i, wrapi(p.j + 1, d.n2), p.k) + f(p.i, wrapi(p.j - 1, d.n2), p.k));
    s += d.w3 * (f(p.i, p.j, wrapi(p.k + 1, d.n3)) + f(p.i, p.j, wrapi(p.k - 1, d.n3)));
    return s;
}
__device__ __forceinline__ int at(const MgDims& d, int i, int j, int k) { return (k * d.n2 + j) * d.n1 + i; }

// x after the first sweep at point t
__device__ __forceinline__ float pre_sweep(const float* __restrict__ b, const MgDims& d, int t, float idiag) {
    const Pt p = point_of(t, d.n1, d.n2);
    if (((p.i + p.j + p.k) & 1) == 0) return b[t] * idiag;
    return (b[t] + idiag * neighbours(d, p, [&](int i, int j, int k) { return b[at(d, i, j, k)]; })) * idiag;
}
// full weighting of the residual at coarse point (I, J, K): sum over the fine points (2I + a, 2J + b, 2K + c),
// a, b, c in {-1, 0, 1}, of w_a w_b w_c (b - A2 x), w_0 = 1/2, w_+-1 = 1/4, red points only
__device__ __forceinline__ float restrict_red(const float* __restrict__ x, const float* __restrict__ b, const MgDims& f,
                                              Pt c) {
    auto res = [&](int a, int bb, int cc) {
        Pt p{wrapi(2 * c.i + a, f.n1), wrapi(2 * c.j + bb, f.n2), wrapi(2 * c.k + cc, f.n3)};
        const int g = at(f, p.i, p.j, p.k);
        return b[g] - (f.diag * x[g] - neighbours(f, p, [&](int i, int j, int k) { return x[at(f, i, j, k)]; }));
    };
    float e = 0.f;
#pragma unroll
    for (int u = -1; u <= 1; u += 2)
#pragma unroll
        for (int v = -1; v <= 1; v += 2) e += res(u, v, 0) + res(u, 0, v) + res(0, u, v);
    return 0.125f * res(0, 0, 0) + 0.03125f * e;
}
// trilinear interpolation of the coarse correction at fine point (i, j, k): fine point 2I + 1 lies between I and I + 1
__device__ __forceinline__ float prolong(const float* __restrict__ xc, const MgDims& c, int i, int j, int k) {
    const int i0 = i >> 1, j0 = j >> 1, k0 = k >> 1;
    const int i1 = (i & 1) ? wrapi(i0 + 1, c.n1) : i0;
    const int j1 = (j & 1) ? wrapi(j0 + 1, c.n2) : j0;
    const int k1 = (k & 1) ? wrapi(k0 + 1, c.n3) : k0;
    return 0.125f * (xc[at(c, i0, j0, k0)] + xc[at(c, i1, j0, k0)] + xc[at(c, i0, j1, k0)] + xc[at(c, i1, j1, k0)] +
                     xc[at(c, i0, j0, k1)] + xc[at(c, i1, j0, k1)] + xc[at(c, i0, j1, k1)] + xc[at(c, i1, j1, k1)]);
}
// point number t of one colour (n1 / 2 per row)
__device__ __forceinline__ Pt colour_point(int t, const MgDims& d, int colour) {
    const int half = d.n1 >> 1, row = t / half;
    Pt p;
    p.k = row / d.n2;
    p.j = row - p.k * d.n2;
    p.i = 2 * (t - row * half) + ((p.j + p.k + colour) & 1);
    return p;
}
__device__ __forceinline__ float post_black(const float* __restrict__ x, const float* __restrict__ b, const MgDims& d,
                                            const float* __restrict__ xc, const MgDims& c, Pt p, float idiag) {
    return (b[at(d, p.i, p.j, p.k)] + neighbours(d, p, [&](int i, int j, int k) {
                return x[at(d, i, j, k)] + prolong(xc, c, i, j, k);
            })) * idiag;
}
__device__ __forceinline__ float post_red(const float* __restrict__ x, const float* __restrict__ b, const MgDims& d,
                                          Pt p, float idiag) {
    return (b[at(d, p.i, p.j, p.k)] + neighbours(d, p, [&](int i, int j, int k) { return x[at(d, i, j, k)]; })) * idiag;
}

__global__ void __launch_bounds__(256) mg_pre_kernel(float* __restrict__ x, const float* __restrict__ b, MgDims d) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < d.n1 * d.n2 * d.n3) x[t] = pre_sweep(b, d, t, 1.f / d.diag);
}
__global__ void __launch_bounds__(128) mg_restrict_kernel(const float* __restrict__ x, const float* __restrict__ b,
                                                          MgDims f, float* __restrict__ bc, MgDims c) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < c.n1 * c.n2 * c.n3) bc[t] = restrict_red(x, b, f, point_of(t, c.n1, c.n2));
}
__global__ void __launch_bounds__(128) mg_black_kernel(float* __restrict__ x, const float* __restrict__ b, MgDims d,
                                                       const float* __restrict__ xc, MgDims c) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (d.n1 >> 1) * d.n2 * d.n3) return;
    const Pt p = colour_point(t, d, 1);
    // black points are written, red ones read
    x[at(d, p.i, p.j, p.k)] = post_black(x, b, d, xc, c, p, 1.f / d.diag);
}
__global__ void __launch_bounds__(256) mg_red_kernel(float* __restrict__ x, const float* __restrict__ b, MgDims d) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (d.n1 >> 1) * d.n2 * d.n3) return;
    const Pt p = colour_point(t, d, 0);
    x[at(d, p.i, p.j, p.k)] = post_red(x, b, d, p, 1.f / d.diag);
}

// The finest level's last half sweep together with what the AAR iteration does with z = M r: the history push
// (X = x - x_prev, F = z - z_prev), and either the Richardson step x += omega z or, when an Anderson step follows, z.
__global__ void __launch_bounds__(256)
mg_finish_kernel(float* __restrict__ z, const float* __restrict__ b, MgDims d, float* __restrict__ x,
                 float* __restrict__ xprev, float* __restrict__ zprev, float* __restrict__ Xs, float* __restrict__ Fs,
                 float omega, int have_prev, int richardson) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= d.n1 * d.n2 * d.n3) return;
    const Pt p = point_of(t, d.n1, d.n2);
    const bool red = ((p.i + p.j + p.k) & 1) == 0;
    const float zt = red ? post_red(z, b, d, p, 1.f / d.diag) : z[t];   // red points of z are written, black ones read
    const float xt = x[t];
    if (have_prev) {
        Xs[t] = xt - xprev[t];
        Fs[t] = zt - zprev[t];
    }
    xprev[t] = xt;
    zprev[t] = zt;
    if (richardson) x[t] = xt + omega * zt;
    else if (red) z[t] = zt;
}

// The small end of the hierarchy (levels of up to a few thousand points) in one CTA, all fields in shared memory: a
// launch per half sweep there costs more than the work.  Levels 0..nl-1 of `A`; the last one is the coarsest grid
// (nl = 1: the coarsest grid alone), solved by K Chebyshev iterations for A2 x = b from x = 0, for the spectrum
// [lmin, lmax] of A2 without its zero eigenvalue (Saad, Iterative Methods for Sparse Linear Systems, Algorithm 12.1).
constexpr int MG_TAIL = 8;
struct MgTail {
    MgDims d[MG_TAIL];
    int off_x[MG_TAIL], off_b[MG_TAIL];   // float offsets into shared memory
    int nl, off_d;                        // off_d: the Chebyshev step of the coarsest grid
    float lmin, lmax;
    int K;
};
__global__ void __launch_bounds__(1024) mg_tail_kernel(float* __restrict__ x, const float* __restrict__ b,
                                                       const __grid_constant__ MgTail A) {
    extern __shared__ float sm[];
    const int nt = blockDim.x, tid = threadIdx.x;
    {
        const int n = A.d[0].n1 * A.d[0].n2 * A.d[0].n3;
        for (int t = tid; t < n; t += nt) sm[A.off_b[0] + t] = b[t];
    }
    __syncthreads();
    for (int l = 0; l + 1 < A.nl; ++l) {
        const MgDims& d = A.d[l];
        const MgDims& c = A.d[l + 1];
        float* xl = sm + A.off_x[l];
        const float* bl = sm + A.off_b[l];
        for (int t = tid; t < d.n1 * d.n2 * d.n3; t += nt) xl[t] = pre_sweep(bl, d, t, 1.f / d.diag);
        __syncthreads();
        for (int t = tid; t < c.n1 * c.n2 * c.n3; t += nt)
            sm[A.off_b[l + 1] + t] = restrict_red(xl, bl, d, point_of(t, c.n1, c.n2));
        __syncthreads();
    }
    {
        const MgDims& d = A.d[A.nl - 1];
        const int n = d.n1 * d.n2 * d.n3;
        float* xs = sm + A.off_x[A.nl - 1];
        const float* bs = sm + A.off_b[A.nl - 1];
        float* ds = sm + A.off_d;
        const float theta = 0.5f * (A.lmax + A.lmin), delta = 0.5f * (A.lmax - A.lmin);
        const float sigma1 = theta / delta;
        for (int p = tid; p < n; p += nt) {
            ds[p] = bs[p] / theta;
            xs[p] = ds[p];
        }
        float rho = 1.f / sigma1;
        for (int it = 1; it < A.K; ++it) {
            __syncthreads();
            const float rho1 = 1.f / (2.f * sigma1 - rho);
            for (int t = tid; t < n; t += nt) {
                const Pt p = point_of(t, d.n1, d.n2);
                const float r = bs[t] - apply_a2(xs, d, p.i, p.j, p.k);
                ds[t] = rho1 * rho * ds[t] + (2.f * rho1 / delta) * r;
            }
            __syncthreads();
            for (int p = tid; p < n; p += nt) xs[p] += ds[p];
            rho = rho1;
        }
        __syncthreads();
    }
    for (int l = A.nl - 2; l >= 0; --l) {
        const MgDims& d = A.d[l];
        const MgDims& c = A.d[l + 1];
        float* xl = sm + A.off_x[l];
        const float* bl = sm + A.off_b[l];
        const float* xc = sm + A.off_x[l + 1];
        const int half = (d.n1 >> 1) * d.n2 * d.n3;
        for (int t = tid; t < half; t += nt) {
            const Pt p = colour_point(t, d, 1);
            xl[at(d, p.i, p.j, p.k)] = post_black(xl, bl, d, xc, c, p, 1.f / d.diag);
        }
        __syncthreads();
        for (int t = tid; t < half; t += nt) {
            const Pt p = colour_point(t, d, 0);
            xl[at(d, p.i, p.j, p.k)] = post_red(xl, bl, d, p, 1.f / d.diag);
        }
        __syncthreads();
    }
    {
        const int n = A.d[0].n1 * A.d[0].n2 * A.d[0].n3;
        for (int t = tid; t < n; t += nt) x[t] = sm[A.off_x[0] + t];
    }
}

MgDims dims_of(const MgLevel& L) {
    MgDims d;
    d.n1 = L.n[0];
    d.n2 = L.n[1];
    d.n3 = L.n[2];
    d.w1 = (float)L.w[0];
    d.w2 = (float)L.w[1];
    d.w3 = (float)L.w[2];
    d.diag = (float)(2.0 * (L.w[0] + L.w[1] + L.w[2]));
    return d;
}

unsigned mg_blocks(long long work, int bs) { return (unsigned)((work + bs - 1) / bs); }

constexpr int MG_COARSE_STOP = 512;    // coarsening stops once a grid has at most this many points
constexpr int MG_COARSE_MAX = 16384;   // largest coarsest grid (x and d in shared memory)
constexpr size_t MG_TAIL_SMEM = 200 * 1024;   // shared memory of the one-CTA end of the hierarchy
// its largest swept level: a tail that takes in a 20^3 level costs 34 us; this one 8.6, plus four launches of 2 to 4 us
constexpr long long MG_TAIL_POINTS = 2048;

}  // namespace

// Level hierarchy of the context's grid: level 0 is the fine grid (its x and b are the V-cycle's
// output and input, supplied per call); each further level halves all three dimensions, until a
// grid has at most MG_COARSE_STOP points or a dimension is odd.  Returns false (no multigrid)
// unless there is at least one coarse level and the coarsest has at most MG_COARSE_MAX points.
bool mg_setup(sdft_ctx* c) {
    c->mg.clear();
    MgLevel L0;
    for (int d = 0; d < 3; ++d) {
        L0.n[d] = c->n[d];
        L0.w[d] = 1.0 / (c->h[d] * c->h[d]);
    }
    L0.np = c->ng;
    std::vector<MgLevel> lv{L0};
    while (true) {
        const MgLevel& f = lv.back();
        if (f.np <= MG_COARSE_STOP) break;
        bool even = true;
        for (int d = 0; d < 3; ++d) even = even && f.n[d] % 2 == 0 && f.n[d] >= 4;
        if (!even) break;
        MgLevel g;
        for (int d = 0; d < 3; ++d) {
            g.n[d] = f.n[d] / 2;
            g.w[d] = f.w[d] / 4.0;
        }
        g.np = (long long)g.n[0] * g.n[1] * g.n[2];
        lv.push_back(g);
    }
    if (lv.size() < 2 || lv.back().np > MG_COARSE_MAX || c->ng >= (1LL << 30)) return false;
    long long tot = 0;
    for (size_t l = 1; l < lv.size(); ++l) tot += 2 * lv[l].np;
    float* buf = (float*)ctx_alloc(c, sizeof(float) * (size_t)tot);
    for (size_t l = 1; l < lv.size(); ++l) {
        lv[l].x = buf;
        lv[l].b = buf + lv[l].np;
        buf += 2 * lv[l].np;
    }
    // coarsest grid: spectrum of the periodic 7-point operator, sum_d 4 w_d sin^2(pi m_d / n_d)
    MgLevel& cl = lv.back();
    double lmax = 0.0, lmin = 1e300;
    for (int d = 0; d < 3; ++d) {
        const double s = std::sin(M_PI * (cl.n[d] / 2) / cl.n[d]);
        lmax += 4.0 * cl.w[d] * s * s;
        const double s1 = std::sin(M_PI / cl.n[d]);
        if (cl.n[d] > 1) lmin = std::min(lmin, 4.0 * cl.w[d] * s1 * s1);
    }
    c->mg_lmin = lmin;
    c->mg_lmax = lmax;
    // iterations for a 1e-1 error bound, 2 q^K <= 1e-1 with q = (sqrt(k) - 1) / (sqrt(k) + 1): as a
    // preconditioner the V-cycle needs no accurate coarse solve (tighter bounds did not reduce the
    // AAR iteration count in a model of the solver)
    const double sk = std::sqrt(lmax / lmin), q = (sk - 1.0) / (sk + 1.0);
    c->mg_coarse_iters = q <= 0.0 ? 1 : std::min(64, std::max(2, (int)std::ceil(std::log(5e-2) / std::log(q))));
    // levels from mg_tail on run in one CTA: x and b of each (x, b and the step of the coarsest) in shared memory
    int first = (int)lv.size() - 1;
    size_t smem = sizeof(float) * 3 * (size_t)cl.np;
    while (first > 1 && (int)lv.size() - first < MG_TAIL && lv[first - 1].np <= MG_TAIL_POINTS &&
           smem + sizeof(float) * 2 * (size_t)lv[first - 1].np <= MG_TAIL_SMEM) {
        --first;
        smem += sizeof(float) * 2 * (size_t)lv[first].np;
    }
    c->mg_tail = first;
    // the attribute belongs to the kernel, not to this context: allow what any context's tail may need
    allow_dynamic_smem(mg_tail_kernel, MG_TAIL_SMEM);
    c->mg = lv;
    return true;
}

namespace {
// the launches of z = M r but for the finest level's last half sweep (mg_finish does it): level 0 uses r and z in
// place of its own b and x
void mg_enqueue(sdft_ctx* c, const float* r, float* z) {
    const int nl = (int)c->mg.size(), tail = c->mg_tail;
    SDFT_REQUIRE(nl >= 2 && tail >= 1, SDFT_ERR_INVALID_ARG, "multigrid V-cycle without a hierarchy");
    auto x = [&](int l) { return l == 0 ? z : c->mg[l].x; };
    auto b = [&](int l) { return l == 0 ? r : (const float*)c->mg[l].b; };
    for (int l = 0; l < tail; ++l) {
        const MgDims d = dims_of(c->mg[l]);
        mg_pre_kernel<<<mg_blocks(c->mg[l].np, 256), 256, 0, c->stream>>>(x(l), b(l), d);
        mg_restrict_kernel<<<mg_blocks(c->mg[l + 1].np, 128), 128, 0, c->stream>>>(x(l), b(l), d, c->mg[l + 1].b,
                                                                                  dims_of(c->mg[l + 1]));
        count_launch(c, 2);
    }
    {
        MgTail A{};
        int off = 0;
        A.nl = nl - tail;
        for (int l = 0; l < A.nl; ++l) {
            const MgLevel& L = c->mg[tail + l];
            A.d[l] = dims_of(L);
            A.off_x[l] = off;
            A.off_b[l] = off + (int)L.np;
            off += 2 * (int)L.np;
        }
        A.off_d = off;
        off += (int)c->mg[nl - 1].np;
        A.lmin = (float)c->mg_lmin;
        A.lmax = (float)c->mg_lmax;
        A.K = c->mg_coarse_iters;
        mg_tail_kernel<<<1, 1024, sizeof(float) * (size_t)off, c->stream>>>(c->mg[tail].x, c->mg[tail].b, A);
        count_launch(c);
    }
    for (int l = tail - 1; l >= 0; --l) {
        const MgDims d = dims_of(c->mg[l]);
        mg_black_kernel<<<mg_blocks(c->mg[l].np / 2, 128), 128, 0, c->stream>>>(x(l), b(l), d, c->mg[l + 1].x,
                                                                               dims_of(c->mg[l + 1]));
        if (l > 0) mg_red_kernel<<<mg_blocks(c->mg[l].np / 2, 256), 256, 0, c->stream>>>(x(l), b(l), d);
        count_launch(c, l > 0 ? 2 : 1);
    }
    SDFT_CUDA(cudaGetLastError());
}
}  // namespace

// r = b + L x and z = M r (but for the last half sweep, see mg_finish) from a zero start.  About ten small launches
// with fixed buffers, so they are captured once into a CUDA graph and replayed; SDFT_MG_GRAPH=0 launches them one by
// one.
void mg_residual_vcycle(sdft_ctx* c, const float* x, const float* b, float* r, float* z) {
    static const bool use_graph = [] {
        const char* env = getenv("SDFT_MG_GRAPH");
        return env == nullptr || atoi(env) != 0;
    }();
    if (!use_graph) {
        laplacian_residual_f32(c, x, b, r);
        mg_enqueue(c, r, z);
        return;
    }
    const float* key[4] = {x, b, r, z};
    if (c->mg_graph && !std::equal(key, key + 4, c->mg_graph_key)) {
        cudaGraphExecDestroy(c->mg_graph);
        c->mg_graph = nullptr;
    }
    if (!c->mg_graph) {
        const uint64_t l0 = c->launches;
        cudaGraph_t graph = nullptr;
        // capture on the private stream (the context's stream may be the legacy default stream)
        if (!c->cap_stream) SDFT_CUDA(cudaStreamCreateWithFlags(&c->cap_stream, cudaStreamNonBlocking));
        cudaStream_t user_stream = c->stream;
        c->stream = c->cap_stream;
        SDFT_CUDA(cudaStreamBeginCapture(c->stream, cudaStreamCaptureModeThreadLocal));
        try {
            laplacian_residual_f32(c, x, b, r);
            mg_enqueue(c, r, z);
        } catch (...) {
            cudaStreamEndCapture(c->stream, &graph);
            if (graph) cudaGraphDestroy(graph);
            c->stream = user_stream;
            throw;
        }
        const cudaError_t ce = cudaStreamEndCapture(c->stream, &graph);
        c->stream = user_stream;
        SDFT_CUDA(ce);
        const cudaError_t ie = cudaGraphInstantiate(&c->mg_graph, graph, 0);
        cudaGraphDestroy(graph);
        SDFT_CUDA(ie);
        c->mg_graph_launches = (int)(c->launches - l0);
        c->launches = l0;
        std::copy(key, key + 4, c->mg_graph_key);
    }
    SDFT_CUDA(cudaGraphLaunch(c->mg_graph, c->stream));
    count_launch(c, c->mg_graph_launches);
}

// the last half sweep of z = M r, the history push and (richardson) the step x += omega z
void mg_finish(sdft_ctx* c, const float* r, float* z, float* x, float* xprev, float* zprev, float* Xs, float* Fs,
               float omega, bool have_prev, bool richardson) {
    mg_finish_kernel<<<mg_blocks(c->ng, 256), 256, 0, c->stream>>>(z, r, dims_of(c->mg[0]), x, xprev, zprev, Xs, Fs,
                                                                  omega, have_prev, richardson);
    SDFT_CUDA(cudaGetLastError());
    count_launch(c);
}

}  // namespace sdft
