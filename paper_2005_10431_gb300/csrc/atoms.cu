// Fields summed over atoms and their periodic images (paper Sec. 2.1 set-up): the Gaussian pseudocharge
// and the superposition of atomic densities on the grid, the radial descriptors of the learned starting
// density, and the self and overlap energies of the pseudocharges with their forces.
//
// The squared distance from a grid point to an image is a sum of three one-axis terms, and a Gaussian a
// product of three one-axis factors, so both come from per-axis tables: entry (atom, image slot m, grid
// index i) of axis d holds the squared displacement d2 of the m-th image of the atom within the cut-off
// of plane i (1e300 where there is none), and exp(-d2 / 2 w^2) or the displacement itself.  A grid kernel then takes one x-row per
// CTA: its threads first test all (atom, z image, y image) candidates against the cut-off, which keeps
// the few that reach the row (ordered, so that sums have a fixed order), and then every thread adds its
// point's x terms for the kept ones.
//
// What bounded these loops before was the FP64 pipe (64 times slower than FP32 on this GPU): every point
// evaluated six FP64 divisions and an exp (or sqrt and cos) for every atom of the cell.
#include "internal.cuh"

#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>

namespace sdft {
namespace {

struct AtomA {
    double pos[3];
    double amp, w, cut;
};

struct AxisTables {
    const double2* t[3];   // [atom][image slot][grid index]: (d2, factor), or (d2, displacement) for direct sums
    int M[3];              // image slots per atom
};

// one thread per (atom, slot, index) of axis d; isolated: the atom itself only
__global__ void axis_table_kernel(const AtomA* __restrict__ at, int natom, int d, int M, int n, double h, double L,
                                  int isolated, int separable, double2* __restrict__ out) {
    const long long total = (long long)natom * M * n;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total; e += (long long)gridDim.x * blockDim.x) {
        const int i = (int)(e % n), m = (int)((e / n) % M), a = (int)(e / ((long long)n * M));
        // the roundings of the displacement are spelled out, so that no contraction changes a direct sum's bits
        const double x = __dmul_rn((double)i, h), p = at[a].pos[d], cut = at[a].cut, w = at[a].w;
        const int lo = isolated ? 0 : (int)ceil((x - p - cut) / L);
        const int hi = isolated ? 0 : (int)floor((x - p + cut) / L);
        const int t = lo + m;
        const bool in = t <= hi;
        const double dx = __fma_rn(-(double)t, L, __dsub_rn(x, p)), d2 = dx * dx;
        out[e] = separable ? make_double2(in ? d2 : 1e300, in ? exp(-d2 / (2.0 * w * w)) : 0.0)
                           : make_double2(in ? d2 : 1e300, dx);
    }
}

// positive doubles order as their bit patterns: the cut-off test stays off the FP64 pipe
__device__ __forceinline__ bool le_bits(double a, double b) {
    return __double_as_longlong(a) <= __double_as_longlong(b);
}

constexpr int ROW_MAXT = 256;

// Row candidates [c0, c0 + blockDim) of all natom * Mz * My: those whose (y, z) distance is within the
// atom's cut-off are kept in shared memory in candidate order.  Returns their number.
struct RowList {
    double w[ROW_MAXT];        // amp * ez * ey (separable), or amp (direct)
    double s[ROW_MAXT];        // dz2 + dy2
    double room[ROW_MAXT];     // cut^2 - s
    double dy[ROW_MAXT], dz[ROW_MAXT];
    int atom[ROW_MAXT];
    int warp_n[ROW_MAXT / 32];
};
__device__ __forceinline__ int gather_row(const AtomA* __restrict__ at, int ncand, int c0, const AxisTables& T, int n2,
                                          int n3, int j, int k, bool separable, RowList& S) {
    const int c = c0 + threadIdx.x;
    bool keep = false;
    double w = 0.0, s = 0.0, room = -1.0;
    double2 y = make_double2(0.0, 0.0), z = y;
    int a = 0;
    if (c < ncand) {
        const int my = c % T.M[1], r = c / T.M[1], mz = r % T.M[2];
        a = r / T.M[2];
        z = T.t[2][((long long)a * T.M[2] + mz) * n3 + k];
        y = T.t[1][((long long)a * T.M[1] + my) * n2 + j];
        const double cut = at[a].cut;
        s = z.x + y.x;
        // a direct sum tests each point's own r^2 in the end: its candidates keep a little slack
        room = cut * cut * (separable ? 1.0 : 1.0 + 1e-12) - s;
        keep = room >= 0.0;
        w = separable ? at[a].amp * (z.y * y.y) : at[a].amp;
    }
    const unsigned ballot = __ballot_sync(0xffffffffu, keep);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __syncthreads();   // the previous list has been consumed
    if (lane == 0) S.warp_n[warp] = __popc(ballot);
    __syncthreads();
    int off = 0, n = 0;
    for (int v = 0; v < (int)(blockDim.x >> 5); ++v) {
        if (v < warp) off += S.warp_n[v];
        n += S.warp_n[v];
    }
    if (keep) {
        const int q = off + __popc(ballot & ((1u << lane) - 1u));
        S.w[q] = w;
        S.s[q] = s;
        S.room[q] = room;
        S.dy[q] = y.y;
        S.dz[q] = z.y;
        S.atom[q] = a;
    }
    __syncthreads();
    return n;
}

// field[g] = sum_a sum_images amp exp(-r^2 / 2 w^2) [r <= cut]; grid: n2 n3 rows, block: n1 rounded up to whole
// warps (at most ROW_MAXT).  SEP: the exponential as a product of the tables' factors; else one exp per point and
// image, each atom's images summed first.  Both fields of the 64-atom cell (80^3): 10.8 ms before, 1.85 ms
// with direct sums, 0.085 ms separable.
template <bool SEP>
__global__ void __launch_bounds__(ROW_MAXT)
atom_field_kernel(const AtomA* __restrict__ at, int natom, const __grid_constant__ AxisTables T, int n1, int n2, int n3,
                  double* __restrict__ field) {
    __shared__ RowList S;
    const int k = blockIdx.x / n2, j = blockIdx.x - k * n2;   // the CTA's row
    const int ncand = natom * T.M[2] * T.M[1];
    for (int i0 = 0; i0 < n1; i0 += blockDim.x) {
        const int i = i0 + threadIdx.x;
        double acc = 0.0, one = 0.0;   // total, and the current atom's sum (direct form)
        int last = -1;
        for (int c0 = 0; c0 < ncand; c0 += blockDim.x) {
            const int n = gather_row(at, ncand, c0, T, n2, n3, j, k, SEP, S);
            if (i < n1)
                for (int q = 0; q < n; ++q) {
                    const int a = S.atom[q];
                    const double2* x = T.t[0] + (long long)a * T.M[0] * n1 + i;
                    const double room = S.room[q], w = S.w[q];
                    if (!SEP && a != last) {
                        acc += one;
                        one = 0.0;
                        last = a;
                    }
                    for (int m = 0; m < T.M[0]; ++m) {
                        const double2 v = x[(long long)m * n1];
                        if (!le_bits(v.x, room)) continue;
                        if (SEP) {
                            acc = fma(w, v.y, acc);
                        } else {
                            const double dx = v.y, dy = S.dy[q], dz = S.dz[q], cut = at[a].cut;
                            const double r2 = __dadd_rn(__fma_rn(dx, dx, __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
                            const double inv = 1.0 / (2.0 * at[a].w * at[a].w);
                            if (r2 <= cut * cut) one = __fma_rn(w, exp(-r2 * inv), one);
                        }
                    }
                }
        }
        if (i < n1) field[(long long)blockIdx.x * n1 + i] = SEP ? acc : acc + one;
    }
}

// Radial descriptors G_q = sum exp(-(r - mu_q)^2 / (2 eta^2)) f_c(r), mu_q = q eta, eta = 6/31, of every
// grid point, in BF16 [ng][32].  The squared distance is FP64; r = hi + lo in two FP32 words (FP32 square root, corrected
// by the FP64 remainder), and the Gaussians' arguments and that of the cut-off function f_c = sin^2(pi (rc - r) / (2 rc))
// keep both words until their last operation.  Against 64-bit sums (cells of 24^3 to 40^3 points) 1.0e-4 to 2.5e-4 of the
// values are rounded to the wrong BF16 neighbour; an FP64 square root and cosine with FP32 distances and exponentials,
// which this replaced, gave 2.5e-4 to 5.9e-4.  Bound by the 32 exponentials per point and atom within 6.5 bohr (issue
// and special function unit).  64-atom cell, 80^3: 4480 -> 152 us; with arguments of one FP32 word and results below
// 2^-126 flushed it took 131 us, misrounded 3.5e-4 to 9.3e-4 and lost half of BF16's subnormal values.
constexpr int NDESC = 32;
constexpr double DESC_RC = 6.5;
// 2^x by the special function unit (2 ulp, as exp2f; results below 2^-126 are kept: BF16 holds values down to 2^-133)
__device__ __forceinline__ float exp2_approx(float x) {
    float y;
    asm("ex2.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// sin^2(pi x), x = (rc - r) / (2 rc) in [0, 1/2], for r = hi + lo: x = xh + xl, sin(pi x) = sin(pi xh) + pi xl cos(pi xh)
// (the cosine, to a few digits, from its Taylor series)
__device__ __forceinline__ float cutoff(float hi, float lo) {
    constexpr float RC = (float)DESC_RC, K = 0.5f / RC, K_LO = (float)(0.5 / DESC_RC - (double)K);
    const float y = RC - hi, yl = ((RC - y) - hi) - lo;
    const float xh = y * K, xl = fmaf(yl, K, fmaf(y, K_LO, fmaf(y, K, -xh)));
    const float x2 = xh * xh, c = fmaf(x2, fmaf(x2, fmaf(x2, -1.33526f, 4.05871f), -4.93480f), 1.f);
    const float s = fmaf(3.14159265f * xl, c, sinpif(xh));
    return s * s;
}
__global__ void __launch_bounds__(ROW_MAXT)
descriptor_row_kernel(const AtomA* __restrict__ at, int natom, const __grid_constant__ AxisTables T, int n1, int n2,
                      int n3, __nv_bfloat16* __restrict__ feat) {
    __shared__ RowList S;
    const int k = blockIdx.x / n2, j = blockIdx.x - k * n2;   // the CTA's row
    const int ncand = natom * T.M[2] * T.M[1];
    for (int i0 = 0; i0 < n1; i0 += blockDim.x) {
        const int i = i0 + threadIdx.x;
        float G[NDESC];
#pragma unroll
        for (int q = 0; q < NDESC; ++q) G[q] = 0.f;
        for (int c0 = 0; c0 < ncand; c0 += blockDim.x) {
            const int n = gather_row(at, ncand, c0, T, n2, n3, j, k, true, S);
            if (i < n1)
                for (int e = 0; e < n; ++e) {
                    const double2* x = T.t[0] + (long long)S.atom[e] * T.M[0] * n1 + i;
                    const double room = S.room[e], s = S.s[e];
                    for (int m = 0; m < T.M[0]; ++m) {
                        const double d2 = x[(long long)m * n1].x;
                        if (!le_bits(d2, room)) continue;
                        const double r2 = d2 + s;
                        const float hi = sqrtf((float)r2);
                        const float lo = hi > 0.f ? (float)fma(-(double)hi, (double)hi, r2) * (0.5f / hi) : 0.f;
                        const float fc = cutoff(hi, lo);
                        // u_q = (r - mu_q) / eta = r 31/6 - q; exp(-u^2 / 2) = 2^(-w^2), w = u sqrt(log2(e) / 2).  r 31/6
                        // as its nearest integer and the rest, so that w is rounded once, relative to itself
                        constexpr float C = 31.f / 6.f, C_LO = (float)(31.0 / 6.0 - (double)C);
                        const float t = hi * C, tl = fmaf(lo, C, fmaf(hi, C_LO, fmaf(hi, C, -t)));
                        constexpr float SK = 0.84932180028801904f;
                        const float ti = rintf(t), wf = ((t - ti) + tl) * SK;
#pragma unroll
                        for (int q = 0; q < NDESC; ++q) {
                            const float w = fmaf(ti - (float)q, SK, wf);
                            G[q] = fmaf(exp2_approx(-w * w), fc, G[q]);
                        }
                    }
                }
        }
        if (i < n1) {
            uint4* o = reinterpret_cast<uint4*>(feat + ((long long)blockIdx.x * n1 + i) * NDESC);
#pragma unroll
            for (int v = 0; v < NDESC / 8; ++v) {
                unsigned b[4];
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    const __nv_bfloat162 h = __floats2bfloat162_rn(G[8 * v + 2 * p], G[8 * v + 2 * p + 1]);
                    b[p] = *reinterpret_cast<const unsigned*>(&h);
                }
                o[v] = make_uint4(b[0], b[1], b[2], b[3]);
            }
        }
    }
}

__global__ void fill_kernel(double* __restrict__ out, double v, long long n) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        out[i] = v;
}

// Overlap correction of the pseudocharges, E_sc = 1/2 sum' Z Z' erfc(d / s) / d over pairs and images within
// rmax, s = sqrt(2 (r^2 + r'^2)), and its gradient with respect to each atom: chunk blockIdx.y of atom
// blockIdx.x's (b, image) list, summed to out[4 (a nchunk + chunk)] = (E, dE/dx, dE/dy, dE/dz).  The host
// loop it replaces took 5 ms for 64 atoms (512 000 candidate images); this takes 92 us.
struct PairAtom {
    double pos[3];
    double Z, r_loc;
};
__global__ void __launch_bounds__(256)
overlap_energy_kernel(const PairAtom* __restrict__ at, int natom, int m1, int m2, int m3, double L1, double L2,
                      double L3, double rmax, double* __restrict__ out) {
    const int a = blockIdx.x;
    const PairAtom A = at[a];
    const int w1 = 2 * m1 + 1, w2 = 2 * m2 + 1, w3 = 2 * m3 + 1;
    const long long total = (long long)natom * w1 * w2 * w3;
    double acc[4] = {0, 0, 0, 0};
    for (long long p = blockIdx.y * (long long)blockDim.x + threadIdx.x; p < total; p += (long long)gridDim.y * blockDim.x) {
        long long r = p;
        const int t2 = (int)(r % w3) - m3;
        r /= w3;
        const int t1 = (int)(r % w2) - m2;
        r /= w2;
        const int t0 = (int)(r % w1) - m1;
        const int b = (int)(r / w1);
        if (b == a && t0 == 0 && t1 == 0 && t2 == 0) continue;
        const PairAtom B = at[b];
        const double v[3] = {A.pos[0] - B.pos[0] - t0 * L1, A.pos[1] - B.pos[1] - t1 * L2, A.pos[2] - B.pos[2] - t2 * L3};
        const double d2 = v[0] * v[0] + v[1] * v[1] + v[2] * v[2];
        if (d2 > rmax * rmax) continue;
        // erfc(q) and exp(-q^2) are below 4e-44 past q = 10: no bit of a sum of larger terms, and such terms alone are
        // no energy
        const double s2 = 2.0 * (A.r_loc * A.r_loc + B.r_loc * B.r_loc);
        if (d2 > 100.0 * s2) continue;
        const double d = sqrt(d2), s = sqrt(s2);
        const double q = d / s, e = erfc(q), zz = A.Z * B.Z;
        acc[0] += 0.5 * zz * e / d;
        if (a != b) {
            const double f = zz * (-2.0 / (s * sqrt(M_PI)) * exp(-q * q) / d - e / d2) / d;
            for (int k = 0; k < 3; ++k) acc[1 + k] += f * v[k];
        }
    }
    __shared__ double sh[4][8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int k = 0; k < 4; ++k) {
        double v = acc[k];
        for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
        if (lane == 0) sh[k][warp] = v;
    }
    __syncthreads();
    if (threadIdx.x < 4) {
        double v = 0.0;
        for (int w = 0; w < 8; ++w) v += sh[threadIdx.x][w];
        out[4 * ((long long)a * gridDim.y + blockIdx.y) + threadIdx.x] = v;
    }
}

// Bytes of the axis tables of natom atoms cut off at `cut`, after their AtomA; M: image slots per atom and axis
size_t axis_bytes(const sdft_ctx* c, double cut, bool iso, int (&M)[3], long long (&size)[3]) {
    long long total = 0;
    for (int d = 0; d < 3; ++d) {
        // at most floor(2 cut / L) + 1 integers lie in an interval of length 2 cut / L
        M[d] = iso ? 1 : (int)std::floor(2.0 * cut / c->L[d]) + 1;
        size[d] = (long long)c->natom * M[d] * c->n[d];
        total += size[d];
    }
    return sizeof(AtomA) * (size_t)c->natom + 256 + sizeof(double2) * (size_t)total;
}

int overlap_chunks(int natom) { return std::max(1, std::min(16, (8 * 152 + natom - 1) / natom)); }
size_t overlap_bytes(int natom) {
    return sizeof(PairAtom) * (size_t)natom + 256 + sizeof(double) * 4 * (size_t)natom * overlap_chunks(natom);
}

// The context's buffer for the tables below: its size follows from the cell, the grid and the species, not from the
// positions, so it is allocated once, at creation, and no later call allocates or releases memory for them.
void reserve_atom_tables(sdft_ctx* c) {
    if (c->atom_tab) return;
    int M[3];
    long long size[3];
    double cut = 0.0;
    for (const sdft_pseudo& s : c->species) cut = std::max(cut, 10.0 * std::max(s.r_loc, s.sad_width));
    size_t bytes = overlap_bytes(c->natom);
    bytes = std::max(bytes, axis_bytes(c, cut, c->opt.boundary == SDFT_BC_DIRICHLET, M, size));
    bytes = std::max(bytes, axis_bytes(c, DESC_RC, false, M, size));
    c->atom_tab = ctx_alloc(c, bytes);
    c->atom_tab_bytes = bytes;
}
// `first` elements of A, then an array of B, in that buffer
template <typename A, typename B>
void atom_tables(sdft_ctx* c, size_t first, A*& a, B*& b) {
    a = reinterpret_cast<A*>(c->atom_tab);
    b = reinterpret_cast<B*>(static_cast<char*>(c->atom_tab) + (sizeof(A) * first + 255) / 256 * 256);
}

inline unsigned nb(long long n) { return (unsigned)std::min<long long>((n + 255) / 256, 152LL * 16); }

// the three axis tables for atoms with positions, widths and cut-offs `at` (device copy in *dat), in the context's buffer
// until the next use of it
struct AxisWork {
    AtomA* dat = nullptr;
    AxisTables T;
    AxisWork(sdft_ctx* c, const std::vector<AtomA>& at, bool iso, bool separable) {
        double cut = 0.0;
        for (const AtomA& a : at) cut = std::max(cut, a.cut);
        long long size[3];
        SDFT_REQUIRE(axis_bytes(c, cut, iso, T.M, size) <= c->atom_tab_bytes, SDFT_ERR_INVALID_ARG, "atom tables too large");
        double2* p = nullptr;
        atom_tables(c, at.size(), dat, p);
        SDFT_CUDA(cudaMemcpyAsync(dat, at.data(), sizeof(AtomA) * at.size(), cudaMemcpyHostToDevice, c->stream));
        for (int d = 0; d < 3; ++d) {
            T.t[d] = p;
            axis_table_kernel<<<nb(size[d]), 256, 0, c->stream>>>(dat, (int)at.size(), d, T.M[d], c->n[d], c->h[d],
                                                                  c->L[d], iso, separable, p);
            p += size[d];
        }
        SDFT_CUDA(cudaGetLastError());
        count_launch(c, 3);
    }
};

std::vector<AtomA> atom_table(const sdft_ctx* c) {
    std::vector<AtomA> at(c->natom);
    for (int a = 0; a < c->natom; ++a)
        for (int d = 0; d < 3; ++d) at[a].pos[d] = c->pos[3 * a + d];
    return at;
}

inline int row_threads(int n1) { return std::min(ROW_MAXT, (n1 + 31) / 32 * 32); }

}  // namespace

// pseudocharge b (atoms cut at 10 r_loc) and SAD density (cut at 10 sad_width, normalised to N_e)
void build_pseudocharge_and_sad(sdft_ctx* c) {
    const int nt = row_threads(c->n[0]);
    const unsigned grid = (unsigned)(c->n[1] * c->n[2]);
    reserve_atom_tables(c);
    // Below 2^15 points the direct sums stay (24^3 points, 2 atoms: 110 us direct, 36 us separable; 40^3 points, 8 atoms:
    // 343 and 49; 48^3 points, 8 atoms: 310 and 50), although they cost more, so that a small cell's fields stay the same
    // bit for bit: an unconverged FP64 SCF started from random orbitals turns a last-bit change of its density into
    // 1e-6 of its energy.  Larger cells take the separable form.
    const bool sep = c->ng >= (1 << 15);
    std::vector<AtomA> at = atom_table(c);
    for (int which = 0; which < 2; ++which) {
        for (int a = 0; a < c->natom; ++a) {
            const sdft_pseudo& s = c->species[c->types[a]];
            const double w = which == 0 ? s.r_loc : s.sad_width;
            at[a].amp = which == 0 ? -s.Z * std::pow(2.0 * M_PI * w * w, -1.5) : s.Z * std::pow(2.0 * M_PI * w * w, -1.5);
            at[a].w = w;
            at[a].cut = 10.0 * w;
        }
        AxisWork W(c, at, c->opt.boundary == SDFT_BC_DIRICHLET, sep);
        double* out = which == 0 ? c->b : c->rho_sad;
        if (sep) atom_field_kernel<true><<<grid, nt, 0, c->stream>>>(W.dat, c->natom, W.T, c->n[0], c->n[1], c->n[2], out);
        else atom_field_kernel<false><<<grid, nt, 0, c->stream>>>(W.dat, c->natom, W.T, c->n[0], c->n[1], c->n[2], out);
        SDFT_CUDA(cudaGetLastError());
        count_launch(c);
    }
    // normalise the SAD density to N_e: sum rho = rho . 1
    double* ones = c->work64;
    fill_kernel<<<nb(c->ng), 256, 0, c->stream>>>(ones, 1.0, c->ng);
    count_launch(c);
    const double* a[1] = {c->rho_sad};
    const double* b[1] = {ones};
    double s = 0.0;
    dots_host(c, 1, a, b, c->ng, &s);
    axpby_dev(c, c->rho_sad, c->rho_sad, 0.0, c->nelec / (c->dV * s), c->ng);
    SDFT_CUDA(cudaGetLastError());
}

// descriptors of every grid point, BF16 [ng][32] (the network's cut-off radius is 6.5 bohr)
void descriptor_field(sdft_ctx* c, void* feat) {
    std::vector<AtomA> at = atom_table(c);
    for (AtomA& a : at) {
        a.amp = 1.0;
        a.w = 1.0;
        a.cut = DESC_RC;
    }
    // images on the periodic lattice whatever the boundary condition, as the network was trained
    AxisWork W(c, at, false, true);
    descriptor_row_kernel<<<(unsigned)(c->n[1] * c->n[2]), row_threads(c->n[0]), 0, c->stream>>>(
        W.dat, c->natom, W.T, c->n[0], c->n[1], c->n[2], reinterpret_cast<__nv_bfloat16*>(feat));
    SDFT_CUDA(cudaGetLastError());
    count_launch(c);
}

// E_self = sum Z^2 / (2 sqrt(pi) r_loc) and the overlap correction with its gradient (host results)
void energy_constants(sdft_ctx* c) {
    const int na = c->natom;
    c->E_self = 0.0;
    std::vector<PairAtom> at(na);
    for (int a = 0; a < na; ++a) {
        const sdft_pseudo& s = c->species[c->types[a]];
        c->E_self += s.Z * s.Z / (2.0 * std::sqrt(M_PI) * s.r_loc);
        at[a] = PairAtom{{c->pos[3 * a], c->pos[3 * a + 1], c->pos[3 * a + 2]}, s.Z, s.r_loc};
    }
    const double rmax = 30.0;
    int m[3];
    for (int d = 0; d < 3; ++d) m[d] = c->opt.boundary == SDFT_BC_DIRICHLET ? 0 : (int)std::ceil(rmax / c->L[d]) + 1;
    const int nchunk = overlap_chunks(na);
    reserve_atom_tables(c);
    PairAtom* dat;
    double* dout;
    atom_tables(c, na, dat, dout);
    SDFT_CUDA(cudaMemcpyAsync(dat, at.data(), sizeof(PairAtom) * na, cudaMemcpyHostToDevice, c->stream));
    overlap_energy_kernel<<<dim3(na, nchunk), 256, 0, c->stream>>>(dat, na, m[0], m[1], m[2], c->L[0], c->L[1], c->L[2],
                                                                   rmax, dout);
    SDFT_CUDA(cudaGetLastError());
    count_launch(c);
    std::vector<double> out((size_t)4 * na * nchunk);
    SDFT_CUDA(cudaMemcpyAsync(out.data(), dout, sizeof(double) * out.size(), cudaMemcpyDeviceToHost, c->stream));
    SDFT_CUDA(cudaStreamSynchronize(c->stream));
    c->E_sc = 0.0;
    c->dEsc.assign(3 * (size_t)na, 0.0);
    for (int a = 0; a < na; ++a)
        for (int k = 0; k < nchunk; ++k) {
            const double* o = &out[4 * ((size_t)a * nchunk + k)];
            c->E_sc += o[0];
            for (int q = 0; q < 3; ++q) c->dEsc[3 * a + q] += o[1 + q];
        }
}

}  // namespace sdft
