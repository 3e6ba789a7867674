// Brick tile of the fused H Y + Chebyshev step, for grids whose blocks fit in L2 (small and medium cells,
// every grid size, Bloch phases, FP32 and FP64):
//
//   Ynext = alpha * (H Y - shift * Y) - beta * Yprev   (see stencil_impl.cuh)
//
// A CTA computes tw x th columns of ZC consecutive planes of one element-column.  Everything it needs from
// Y is loaded up front with all loads in flight: each thread's column of ZC + 12 planes into registers, the
// x and y halo of the ZC planes and the columns themselves into shared memory; after one barrier the ZC
// planes are computed without any further wait on Y.  The column tile instead marches through the planes
// with one barrier and one memory latency per plane, which a small grid cannot hide: with 24 to 48 points an
// edge there are one or two CTAs per SM, each 24 to 48 steps of latency long (plus 12 planes of warm-up per
// z chunk).  Bricks are ZC planes long, so the same grid gives several times the CTAs, and tw x th is chosen
// per grid so that few threads fall outside it (the column tile's 32-wide rows leave 42 % of the threads
// idle at 37 points).  The price is more halo per point, which L2 serves.
// The row stride tw + 16 makes consecutive tile rows continue the bank sequence, so a warp that straddles
// rows reads 32 consecutive columns' banks without conflicts.
// Sums are formed in the column tile's order: real blocks get the same bits.  (Bloch blocks round the product of two
// phase factors differently at the cell's edges: 1e-16 of the largest value in FP64, 6e-8 in FP32.)
// Measured, column tile -> brick, us per step (kernel time): 24^3, FP64, 8 columns 87 -> 12; 37 x 41 x 45, FP32, 20 columns 31 -> 15;
// 40^3, Bloch, 20 columns 59 -> 25; 48^3, 40 columns 66 -> 35; 32 cells of 24 to 48 points in one launch 427 -> 310.
// Bound by issue and shared-memory reads of one tile at a time (two CTAs per SM).  Staging V_eff and the KB slots in
// shared memory as well was slower (15 -> 20, 25 -> 36, 310 -> 385).
#pragma once
#include "stencil_impl.cuh"

namespace sdft {
namespace {

constexpr int BRICK_NT = 256;   // at most tw * th threads
constexpr size_t BRICK_SMEM_MAX = 110 * 1024;   // tile and KB coefficients of a CTA, two CTAs per SM

struct BrickTile {
    int tw, th;          // columns per CTA
    int tiles_x, tiles_y;
};

// The split of an n1 x n2 plane into equal tiles of at most BRICK_NT columns that costs least: thread slots
// (whole warps) plus a third per halo element of a plane.  tw stays at or below 64 so that the shared-memory
// tile of an 8-plane FP32 brick fits four to a SM.
inline BrickTile brick_tile(int n1, int n2) {
    BrickTile best{0, 0, 0, 0};
    double best_cost = 1e300;
    for (int kx = (n1 + 63) / 64; kx <= (n1 + 7) / 8; ++kx) {
        const int tw = (n1 + kx - 1) / kx;
        const int thmax = std::max(1, std::min(n2, BRICK_NT / tw));
        const int ky = (n2 + thmax - 1) / thmax;
        const int th = (n2 + ky - 1) / ky;
        const double cost = (double)kx * ky * ((tw * th + 31) / 32 * 32 + 4.0 * (tw + th));
        if (cost < best_cost) {
            best_cost = cost;
            best = BrickTile{tw, th, (n1 + tw - 1) / tw, (n2 + th - 1) / th};
        }
    }
    return best;
}

// shared memory: ZC halo'd planes, then the KB coefficients of the column
template <typename E>
inline size_t brick_smem(const BrickTile& t, int zc, int natom) {
    return sizeof(E) * ((size_t)zc * (t.th + 2 * FD_RADIUS) * (t.tw + 16) + natom);
}

// x in [-6, 2 n) -> [0, n), t = number of edges crossed (tiles start inside the grid and end less than n past it)
__device__ __forceinline__ int wrap_once(int x, int n, int& t) {
    t = x < 0 ? -1 : (x >= n ? 1 : 0);
    return x - t * n;
}

// Body for tile (bx, by), planes [z0, min(z0 + ZC, n3)) of element-column col.
template <typename E, bool CPLX, int ZC, bool PREV, bool KB>
__device__ __forceinline__ void brick_body(const E* __restrict__ Y, const E* __restrict__ Yprev, E* __restrict__ Ynext,
                                           const typename Elem<E>::S* __restrict__ V, const E* __restrict__ C,
                                           const int* __restrict__ patom, const void* __restrict__ pval,
                                           const int nslot, const StepArgs<typename Elem<E>::S>& A,
                                           const typename Elem<E>::S alpha, const typename Elem<E>::S beta,
                                           const int tw, const int th, const int bx, const int by, const int z0,
                                           const int col) {
    using S = typename Elem<E>::S;
    using KV = typename std::conditional<CPLX, E, S>::type;
    constexpr int R = FD_RADIUS;
    constexpr int SP = sizeof(KV) <= 4 ? 3 : 2;   // KB slots fetched a plane ahead (further ones at their use)
    extern __shared__ __align__(16) unsigned char dyn_smem[];
    E* tile = reinterpret_cast<E*>(dyn_smem);
    const int RS = tw + 16, PS = (th + 2 * R) * RS;   // row and plane stride of the staged tile
    E* Cs = tile + ZC * PS;
    const int tid = threadIdx.x;
    const int ty = tid / tw, tx = tid - ty * tw;
    const int x0 = bx * tw, y0 = by * th;
    const int gx = x0 + tx, gy = y0 + ty;
    const bool inside = ty < th;
    const bool valid = inside && gx < A.n1 && gy < A.n2;
    const int nz = min(ZC, A.n3 - z0);
    const unsigned plane = (unsigned)(A.n1 * A.n2);   // offsets within a column fit 32 bits (brick_ok)
    const E* __restrict__ Yc = Y + (long long)col * A.ng;
    const E* __restrict__ Pc = Yprev + (long long)col * A.ng;
    const KV* __restrict__ pv = reinterpret_cast<const KV*>(pval);
    auto phase = [&](int txw, int tyw) {   // Bloch factor of a column tx, ty periods away
        E ph = eone<E>();
        if constexpr (CPLX) {
            if (txw) ph = apply_phase<E, S>(ph, txw, A.phr[0], A.phi[0]);
            if (tyw) ph = apply_phase<E, S>(ph, tyw, A.phr[1], A.phi[1]);
        }
        return ph;
    };

    // own column: planes z0 - R .. z0 + ZC + R - 1 (wrapped; columns past the grid edge hold the wrapped
    // column, which is their neighbours' halo)
    E q[ZC + 2 * R];
    if (inside) {
        int txw, tyw;
        const int wx = wrap_once(gx, A.n1, txw), wy = wrap_once(gy, A.n2, tyw);
        const unsigned base = (unsigned)(wy * A.n1 + wx);
        int tz = z0 - R < 0 ? -1 : 0, wz = z0 - R - tz * A.n3;
        unsigned off = wz * plane + base;
#pragma unroll
        for (int s = 0; s < ZC + 2 * R; ++s) {
            q[s] = Yc[off];
            if constexpr (CPLX) {
                if (tz) q[s] = apply_phase<E, S>(q[s], tz, A.phr[2], A.phi[2]);
            }
            off += plane;
            if (++wz == A.n3) {
                wz = 0;
                ++tz;
                off = base;
            }
        }
        if constexpr (CPLX) {
            if (txw | tyw) {
                const E ph = phase(txw, tyw);
#pragma unroll
                for (int s = 0; s < ZC + 2 * R; ++s) q[s] = cmul(q[s], ph);
            }
        }
    }
    // operands of one plane of the own column, fetched a plane ahead of their use
    struct Ops {
        S v;
        E prev;
        int at[SP];
        KV kv[SP];
    };
    const unsigned g0 = (unsigned)z0 * plane + (unsigned)(gy * A.n1 + gx);
    auto fetch = [&](int p, Ops& o) {
        const unsigned g = g0 + p * plane;
        o.v = V[g];
        if (PREV) o.prev = Pc[g];
        if (KB) {
#pragma unroll
            for (int s = 0; s < SP; ++s)
                if (s < nslot) {
                    o.at[s] = patom[s * A.ng + g];
                    o.kv[s] = pv[s * A.ng + g];
                }
        }
    };
    Ops cur, nxt;
    if (valid) fetch(0, cur);
    // halo of the ZC planes: th rows of R + R columns, then R + R rows of tw columns
    const int nhx = 2 * R * th, nh = nhx + 2 * R * tw;
    for (int i = tid; i < nh; i += blockDim.x) {
        int ly, lx;
        if (i < nhx) {
            ly = i / (2 * R);
            lx = i - ly * (2 * R);
            lx = lx < R ? lx : tw + lx;
            ly += R;
        } else {
            const int k = i - nhx;
            ly = k / tw;
            lx = R + k - ly * tw;
            ly = ly < R ? ly : th + ly;
        }
        int txw, tyw;
        const int wx = wrap_once(x0 - R + lx, A.n1, txw), wy = wrap_once(y0 - R + ly, A.n2, tyw);
        const unsigned base = (unsigned)z0 * plane + (unsigned)(wy * A.n1 + wx);
        E h[ZC];
#pragma unroll
        for (int p = 0; p < ZC; ++p) h[p] = Yc[base + min(p, nz - 1) * plane];
        if constexpr (CPLX) {
            if (txw | tyw) {
                const E ph = phase(txw, tyw);
#pragma unroll
                for (int p = 0; p < ZC; ++p) h[p] = cmul(h[p], ph);
            }
        }
#pragma unroll
        for (int p = 0; p < ZC; ++p) tile[p * PS + ly * RS + lx] = h[p];
    }
    if (KB)
        for (int i = tid; i < A.natom; i += blockDim.x) Cs[i] = C[(long long)col * A.natom + i];
    if (inside) {
#pragma unroll
        for (int p = 0; p < ZC; ++p) tile[p * PS + (R + ty) * RS + R + tx] = q[R + p];
    }
    __syncthreads();
    if (!valid) return;
    E* __restrict__ Zc = Ynext + (long long)col * A.ng;
#pragma unroll
    for (int p = 0; p < ZC; ++p) {
        if (p < nz) {
            if (p + 1 < nz) fetch(p + 1, nxt);
            const unsigned g = g0 + p * plane;
            const E* T = tile + p * PS + (R + ty) * RS + R + tx;
            const E center = q[R + p];
            E az = efma(A.c0, center, ezero<E>()), ax = ezero<E>(), ay = ezero<E>();
#pragma unroll
            for (int r = 1; r <= R; ++r) {
                az = efma(A.cz[r], eadd(q[R + p + r], q[R + p - r]), az);
                ax = efma(A.cx[r], eadd(T[r], T[-r]), ax);
                ay = efma(A.cy[r], eadd(T[r * RS], T[-r * RS]), ay);
            }
            E acc = eadd(az, eadd(ax, ay));
            acc = efma(cur.v, center, acc);
            if (KB) {
#pragma unroll
                for (int s = 0; s < SP; ++s)
                    if (s < nslot && cur.at[s] >= 0) {
                        if constexpr (CPLX) acc = eadd(acc, cmul(cur.kv[s], Cs[cur.at[s]]));
                        else acc = efma(cur.kv[s], Cs[cur.at[s]], acc);
                    }
                if (nslot > SP && cur.at[SP - 1] >= 0)   // slots are filled in order and padded with atom -1
                    for (int s = SP; s < nslot; ++s) {
                        const int a = __ldg(patom + s * A.ng + g);
                        if (a < 0) break;
                        if constexpr (CPLX) acc = eadd(acc, cmul(pv[s * A.ng + g], Cs[a]));
                        else acc = efma(pv[s * A.ng + g], Cs[a], acc);
                    }
            }
            E out = efma(alpha, efma(-A.shift, center, acc), ezero<E>());
            if (PREV) out = efma(-beta, cur.prev, out);
            Zc[g] = out;
            cur = nxt;
        }
    }
}

// grid: (tiles_x * tiles_y, z chunks, columns)
template <typename E, bool CPLX, int ZC, int MINB, bool PREV, bool KB>
__global__ void __launch_bounds__(BRICK_NT, MINB)
brick_kernel(const E* __restrict__ Y, const E* __restrict__ Yprev, E* __restrict__ Ynext,
             const typename Elem<E>::S* __restrict__ V, const E* __restrict__ C, const int* __restrict__ patom,
             const void* __restrict__ pval, const int nslot, const int tw, const int th, const int tiles_x,
             const __grid_constant__ StepArgs<typename Elem<E>::S> A) {
    const int by = blockIdx.x / tiles_x, bx = blockIdx.x - by * tiles_x;
    brick_body<E, CPLX, ZC, PREV, KB>(Y, Yprev, Ynext, V, C, patom, pval, nslot, A, A.alpha, A.beta, tw, th, bx, by,
                                      blockIdx.y * ZC,
                                      blockIdx.z);
}

// Column counts and plane counts above the grid limits, columns past 32-bit offsets and KB coefficients that do
// not fit beside the tile are not taken (callers fall back to the column tile).
template <typename E, int ZC>
bool brick_ok(const sdft_ctx* c, int ncolE) {
    return ncolE > 0 && ncolE <= 65535 && (c->n[2] + ZC - 1) / ZC <= 65535 && c->ng < (1LL << 31) &&
           c->opt.boundary == SDFT_BC_PERIODIC &&
           brick_smem<E>(brick_tile(c->n[0], c->n[1]), ZC, c->natom) <= BRICK_SMEM_MAX;
}

template <typename E, bool CPLX, int ZC, int MINB>
void launch_brick(sdft_ctx* c, int kpt, const E* Y, const E* Yprev, E* Ynext, int ncolE,
                  const typename Elem<E>::S* V, const E* kbC, double alpha, double beta, double shift, bool kin,
                  bool timed) {
    using S = typename Elem<E>::S;
    SDFT_REQUIRE(kin && V != nullptr, SDFT_ERR_INVALID_ARG, "brick stencil tile needs V and the kinetic term");
    SDFT_REQUIRE((brick_ok<E, ZC>(c, ncolE)), SDFT_ERR_INVALID_ARG, "brick stencil tile does not fit");
    const BrickTile t = brick_tile(c->n[0], c->n[1]);
    const int nzc = (c->n[2] + ZC - 1) / ZC;
    StepArgs<S> A = make_args<S>(c, kpt, alpha, beta, shift, ZC, nzc);
    const dim3 grid(t.tiles_x * t.tiles_y, nzc, ncolE);
    const int nt = (t.tw * t.th + 31) / 32 * 32;
    const KBTables& kb = c->kb[kpt];
    const void* pval = std::is_same<S, float>::value ? (const void*)kb.pval32 : (const void*)kb.pval64;
    const size_t dsm = brick_smem<E>(t, ZC, c->natom);
    const bool prev = Yprev != nullptr, haskb = kbC != nullptr && kb.S > 0;
    ScopedTimer timer(timed ? c : nullptr, sizeof(S) == 8 ? SDFT_K_STENCIL64 : SDFT_K_STENCIL,
                      (double)ncolE * (double)c->ng * sizeof(E) * (prev ? 3.0 : 2.0));
    auto launch = [&](auto kfn) {
        if (dsm > 48 * 1024) allow_dynamic_smem(kfn, BRICK_SMEM_MAX);
        kfn<<<grid, nt, dsm, c->stream>>>(Y, Yprev, Ynext, V, kbC, kb.patom, pval, kb.S, t.tw, t.th, t.tiles_x, A);
    };
    if (prev && haskb) launch(brick_kernel<E, CPLX, ZC, MINB, true, true>);
    else if (!prev && haskb) launch(brick_kernel<E, CPLX, ZC, MINB, false, true>);
    else if (prev) launch(brick_kernel<E, CPLX, ZC, MINB, true, false>);
    else launch(brick_kernel<E, CPLX, ZC, MINB, false, false>);
    SDFT_CUDA(cudaGetLastError());
    count_launch(c);
}

}  // namespace
}  // namespace sdft
