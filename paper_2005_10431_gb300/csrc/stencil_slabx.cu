// Slab tile of the fused H Y + Chebyshev step for FP32 real blocks on any grid with even n1:
//
//   Ynext = alpha * (H Y - shift * Y) - beta * Yprev      (see stencil_impl.cuh)
//
// The schedule is that of the slab tiles in stencil_tma.cu (a CTA marches along z with TY whole x-rows, a producer warp
// feeds a ring of stages, z-neighbours in a register queue).  Those are bound by the shared-memory pipe: 19 16-byte
// reads for a thread's two points, 12 of them y-neighbours.  Here a thread owns the same two x-points of two
// neighbouring rows of one orbital pair, so that 12 halo rows and its own registers hold the y-neighbours of four
// points (28 reads for four points).  Every halo value is added to both rows as it is read: keeping the values for the
// second row spilled 2.5 KB per thread and cost twice the time.  Row length, TY and the number of staged KB slots are launch
// parameters:
//   * rows are contiguous in memory, so a stage is fed by untiled bulk copies: the TY + 12 halo'd rows in one run, or
//     more where the tile crosses the periodic y edge.  A ragged last slab copies its own rows only and does not
//     store the others;
//   * V_eff and KB rows (4-byte values, n1 even) start on an 8-byte boundary: their copies start up to two values early,
//     and the reader skips them;
//   * KB slots past the staged ones are read from L2 by the few points that have them.
//   * the diagonal of the kinetic term and V_eff are added last.  Added first, as the largest term, they set the rounding
//     of the 24 sums that follow: H X was off by 1.27e-7 (root mean square, relative), 0.59e-7 now, column tile 0.80e-7.
// TY is what 320 compute threads hold (11 warps of 168 registers): 2 floor(640 / n1) rows, evened out over the slabs.
// Measured, us per step (best of the other tiles -> this one): 82 x 82 x 76, 176 columns 706 -> 358 (at 100 % of the
// copy bandwidth 160); 96^3, 300 columns 1600 -> 915 (471); 64 x 60 x 60, 66 columns 115 -> 63 (27).  Latency of the few
// warps bounds it (issue slots 47 %, shared-memory pipe 60 %, DRAM 49 %): for n1 = 80 and 120 the slab tiles with
// compiled-in row lengths stay (294 and 304, 2605 and 3079).  One row a thread instead of two took 402, 1084 and 68.
#include "internal.cuh"
#include "stencil_ptx.cuh"

#include <algorithm>

namespace sdft {

int sm_count();   // stencil_tma.cu

namespace {

constexpr int R = FD_RADIUS;
constexpr int SX_PFD = 10;              // planes between a stage's copies and the L2 prefetch issued with them
constexpr int SX_MAXD = 6;              // stages
constexpr size_t SX_RING = 225 * 1024;
constexpr size_t SX_TAIL = 16 * SX_MAXD + 128;   // barriers and the ring's alignment
constexpr int SX_COMP = 320;            // compute threads at most
constexpr int SX_MAXT = SX_COMP + 32;

struct SlabxArgs {
    float2 cx[R + 1], cy[R + 1], cz[R + 1];   // both lanes of a packed multiplier
    float2 alpha, mbeta;                // mbeta = -beta
    float c0;                           // diagonal of the kinetic term, less the shift
    int n1, n2, n3, ty, nslab, ncolE, natom, nslot, nst, depth;
    unsigned off_q, off_prev, off_v, off_ka, off_kv, off_c, kbytes, sstride;   // byte offsets in a stage; bytes per KB slot
    long long ng;
    unsigned vmis;                      // V's offset from a 16-byte boundary, in values
    unsigned ngl;                       // ng modulo 2^32
    int total, per_cta;                 // (pair group, plane) units of a slab, and of a CTA
};

// KB sums of the point pairs at byte offset v of the stage's 4-byte rows and one row further, from the staged slots.
// Slots fill in order, so a warp whose points all have an empty slot has no later one.
__device__ __forceinline__ void slabx_kb(uint32_t st, uint32_t cg, uint32_t v, uint32_t vrow, unsigned g0, const SlabxArgs& A,
                                         float2& s00, float2& s01, float2& s10, float2& s11) {
    const float2 zero = make_float2(0.f, 0.f);
    for (int k = 0; k < A.nst; ++k) {
        const uint32_t a = (uint32_t)k * A.kbytes + (((unsigned)k * A.ngl + g0) & 3u) * 4u + v;
        const int2 ka = lds64i(st + A.off_ka + a), kb = lds64i(st + A.off_ka + a + vrow);
        const unsigned na = (unsigned)A.natom;
        const bool v0 = (unsigned)ka.x < na, v1 = (unsigned)ka.y < na, v2 = (unsigned)kb.x < na, v3 = (unsigned)kb.y < na;
        if (!__any_sync(0xffffffffu, v0 || v1 || v2 || v3)) break;
        const float2 wa = lds64(st + A.off_kv + a), wb = lds64(st + A.off_kv + a + vrow);
        const float2 c0 = lds64(cg + (v0 ? (uint32_t)ka.x * 8u : 0u)), c1 = lds64(cg + (v1 ? (uint32_t)ka.y * 8u : 0u));
        const float2 c2 = lds64(cg + (v2 ? (uint32_t)kb.x * 8u : 0u)), c3 = lds64(cg + (v3 ? (uint32_t)kb.y * 8u : 0u));
        s00 = fma2(wa.x, v0 ? c0 : zero, s00);
        s01 = fma2(wa.y, v1 ? c1 : zero, s01);
        s10 = fma2(wb.x, v2 ? c2 : zero, s10);
        s11 = fma2(wb.y, v3 ? c3 : zero, s11);
    }
}
// the slots past the staged ones, from global memory
__device__ __forceinline__ void slabx_kb_far(uint32_t cg, unsigned g, const int* __restrict__ patom,
                                             const float* __restrict__ pval, const SlabxArgs& A, float2& s0, float2& s1) {
    for (int k = A.nst; k < A.nslot; ++k) {
        const int2 ka = __ldg(reinterpret_cast<const int2*>(patom + k * A.ng + g));
        if (ka.x < 0 && ka.y < 0) break;
        const float2 kv = __ldg(reinterpret_cast<const float2*>(pval + k * A.ng + g));
        if (ka.x >= 0) s0 = fma2(kv.x, lds64(cg + (uint32_t)ka.x * 8u), s0);
        if (ka.y >= 0) s1 = fma2(kv.y, lds64(cg + (uint32_t)ka.y * 8u), s1);
    }
}
// x-neighbours of the point pair m: points x-6 .. x+7 of the row at T from six 16-byte reads
__device__ __forceinline__ void slabx_x(uint32_t T, const int (&xc)[6], const SlabxArgs& A, float4 m, float2& s0, float2& s1) {
    const float4 L2 = lds128(T + xc[2]), R0 = lds128(T + xc[3]);
    s0 = fma2v(A.cx[1], add2(hi2(L2), hi2(m)), s0);
    s0 = fma2v(A.cx[2], add2(lo2(L2), lo2(R0)), s0);
    s1 = fma2v(A.cx[1], add2(lo2(m), lo2(R0)), s1);
    s1 = fma2v(A.cx[2], add2(hi2(L2), hi2(R0)), s1);
    const float4 L1 = lds128(T + xc[1]), R1 = lds128(T + xc[4]);
    s0 = fma2v(A.cx[3], add2(hi2(L1), hi2(R0)), s0);
    s0 = fma2v(A.cx[4], add2(lo2(L1), lo2(R1)), s0);
    s1 = fma2v(A.cx[3], add2(lo2(L2), lo2(R1)), s1);
    s1 = fma2v(A.cx[4], add2(hi2(L1), hi2(R1)), s1);
    const float4 L0 = lds128(T + xc[0]), R2 = lds128(T + xc[5]);
    s0 = fma2v(A.cx[5], add2(hi2(L0), hi2(R1)), s0);
    s0 = fma2v(A.cx[6], add2(lo2(L0), lo2(R2)), s0);
    s1 = fma2v(A.cx[5], add2(lo2(L1), lo2(R2)), s1);
    s1 = fma2v(A.cx[6], add2(hi2(L0), hi2(R2)), s1);
}

template <bool PREV, bool KB>
__global__ void __launch_bounds__(SX_MAXT, 1)
cheb_slabx_kernel(const float2* __restrict__ Y, const float2* __restrict__ Yprev, float2* __restrict__ Ynext,
                  const float* __restrict__ V, const float2* __restrict__ C, const int* __restrict__ patom,
                  const float* __restrict__ pval, const __grid_constant__ SlabxArgs A, int* __restrict__ err) {
    constexpr int QN = 2 * R + 1;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    unsigned char* smem = smem_raw + ((128u - ((unsigned)__cvta_generic_to_shared(smem_raw) & 127u)) & 127u);
    const int D = A.depth, n1 = A.n1, n2 = A.n2, n3 = A.n3, TY = A.ty;
    const uint32_t rowb = (uint32_t)n1 * 8u, tileb = (uint32_t)(TY + 2 * R) * rowb;
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + (size_t)A.sstride * D);
    uint64_t* empty = full + SX_MAXD;
    const int tid = threadIdx.x, ncomp = blockDim.x - 32;
    const int slab = blockIdx.x % A.nslab;
    const int fbeg = (blockIdx.x / A.nslab) * A.per_cta, fend = min(A.total, fbeg + A.per_cta);
    if (fbeg >= fend) return;   // whole CTA, before any barrier
    const unsigned plane = (unsigned)(n1 * n2);
    const int y0 = slab * TY;
    if (tid == ncomp) {
        for (int s = 0; s < D; ++s) {
            mb_init(&full[s], 1);
            mb_init(&empty[s], ncomp / 32);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    bool ok = true;
    int issued = 0;   // planes whose copies the producer lane has issued
    if (tid >= ncomp) {
        // ---------------- producer warp: one lane issues every copy ----------------
        if (tid == ncomp) {
            const int rows = min(TY, n2 - y0);   // rows of the slab inside the grid
            int slot = 0;
            uint32_t par = 1;
            for (int f = fbeg; f < fend && ok;) {
                const int col = f / n3, z0 = f - col * n3, z1 = min(n3, z0 + (fend - f));
                const float2* Yc = Y + (long long)col * A.ng;
                const float2* Pc = Yprev + (long long)col * A.ng;
                const long long e0 = (long long)col * A.natom;
                const int o = (int)(e0 & 1);
                const uint32_t kcb = KB ? (uint32_t)((o + A.natom + 1) & ~1) * 8u : 0u;
                for (int z = z0; z < z1; ++z) {
                    if (issued >= D && !mb_wait(&empty[slot], par)) {
                        ok = false;
                        break;
                    }
                    unsigned char* st = smem + (size_t)slot * A.sstride;
                    // 4-byte rows: offset of the slab's first value, the copy's start on a 16-byte boundary
                    const unsigned g0 = (unsigned)z * plane + (unsigned)(y0 * n1), sh = (g0 + A.vmis) & 3u;
                    const uint32_t vb = ((uint32_t)(rows * n1) + sh) * 4u, vb16 = (vb + 15u) & ~15u;
                    uint32_t bytes = tileb + (uint32_t)TY * rowb + (PREV ? (uint32_t)rows * rowb : 0u) + vb16 + kcb;
                    if (KB)
                        for (int k = 0; k < A.nst; ++k) {
                            const uint32_t s = (uint32_t)((k * A.ng + g0) & 3);
                            bytes += 2u * ((((uint32_t)(rows * n1) + s) * 4u + 15u) & ~15u);
                        }
                    mb_expect_tx(&full[slot], bytes);
                    int zq = z + R;
                    while (zq >= n3) zq -= n3;
                    const float2* row0 = Yc + (size_t)z * plane;
                    int y = y0 - R;
                    while (y < 0) y += n2;
                    for (int r = 0; r < TY + 2 * R;) {   // contiguous runs of rows up to the periodic edge
                        const int len = min(n2 - y, TY + 2 * R - r);
                        bulk_copy(st + (size_t)r * rowb, row0 + (size_t)y * n1, (uint32_t)len * rowb, &full[slot]);
                        r += len;
                        y = 0;
                    }
                    y = y0;
                    for (int r = 0; r < TY;) {   // all TY rows: the last stored row's neighbour may be row 0
                        const int len = min(n2 - y, TY - r);
                        bulk_copy(st + A.off_q + (size_t)r * rowb, Yc + (size_t)zq * plane + (size_t)y * n1,
                                  (uint32_t)len * rowb, &full[slot]);
                        r += len;
                        y = 0;
                    }
                    if (PREV)
                        bulk_copy(st + A.off_prev, Pc + (size_t)z * plane + (size_t)y0 * n1, (uint32_t)rows * rowb, &full[slot]);
                    bulk_copy(st + A.off_v, V + g0 - sh, vb16, &full[slot]);
                    if (KB) {
                        for (int k = 0; k < A.nst; ++k) {
                            const long long gk = k * A.ng + g0;
                            const uint32_t s = (uint32_t)(gk & 3), b16 = (((uint32_t)(rows * n1) + s) * 4u + 15u) & ~15u;
                            bulk_copy(st + A.off_ka + (size_t)k * A.kbytes, patom + (gk - s), b16, &full[slot]);
                            bulk_copy(st + A.off_kv + (size_t)k * A.kbytes, pval + (gk - s), b16, &full[slot]);
                        }
                        bulk_copy(st + A.off_c, C + (e0 - o), kcb, &full[slot]);
                    }
                    ++issued;
                    if (++slot == D) {
                        slot = 0;
                        par ^= 1u;
                    }
                    const int zp = z + SX_PFD;
                    if (zp < z1) {
                        const size_t off = (size_t)zp * plane + (size_t)y0 * n1;
                        prefetch_bulk(Yc + off, (uint32_t)rows * rowb);
                        if (PREV) prefetch_bulk(Pc + off, (uint32_t)rows * rowb);
                    }
                }
                f += z1 - z0;
            }
            if (!ok) atomicExch(err, 1);
        }
    } else {
        // ---------------- compute warps: two x-points of two rows ----------------
        const int hx = n1 >> 1;
        int ty = tid / hx, tx = tid - ty * hx;
        const bool act = 2 * ty < TY;
        if (!act) ty = tx = 0;   // threads past the last row repeat the first one's work and store nothing
        ty *= 2;
        const int gx = 2 * tx;
        const bool st0 = act && y0 + ty < n2, st1 = act && ty + 1 < TY && y0 + ty + 1 < n2;
        int xc[6];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const int l = gx - 6 + 2 * k, r = gx + 2 + 2 * k;
            xc[k] = (l < 0 ? l + n1 : l) * 8;
            xc[3 + k] = (r >= n1 ? r - n1 : r) * 8;
        }
        const uint32_t ring = s32(smem);
        const uint32_t own = (uint32_t)ty * rowb + (uint32_t)gx * 8u;      // within the Q and PREV rows
        const uint32_t vown = (uint32_t)(ty * n1 + gx) * 4u, vrow = (uint32_t)n1 * 4u;   // within the 4-byte rows
        const int yr0 = (y0 + ty) % n2, yr1 = (y0 + ty + 1) % n2;
        const unsigned gxy = (unsigned)(yr0 * n1 + gx), gxy1 = (unsigned)(yr1 * n1 + gx);
        int slot = 0;
        uint32_t par = 0;
        for (int f = fbeg; f < fend && ok;) {
            const int col = f / n3, z0 = f - col * n3, z1 = min(n3, z0 + (fend - f));
            const float2* __restrict__ Yg = Y + (long long)col * A.ng;
            float2* __restrict__ Zg = Ynext + (long long)col * A.ng;
            const uint32_t cofs = A.off_c + 8u * (uint32_t)(((long long)col * A.natom) & 1);
            float4 q0[QN], q1[QN];
            {   // planes z0 - R .. z0 + R - 1; each stage then brings plane z + R
                int wz = z0 - R < 0 ? z0 - R + n3 : z0 - R;
#pragma unroll
                for (int s = 0; s < 2 * R; ++s) {
                    const float2* r = Yg + (size_t)wz * plane;
                    q0[s] = *reinterpret_cast<const float4*>(r + gxy);
                    q1[s] = *reinterpret_cast<const float4*>(r + gxy1);
                    if (++wz == n3) wz = 0;
                }
            }
            for (int zb = z0; zb < z1 && ok; zb += QN) {
#pragma unroll
                for (int ph = 0; ph < QN; ++ph) {
                    const int z = zb + ph;
                    if (z < z1 && ok) {
                        // a warp-uniform outcome keeps the __syncwarp below convergent
                        if (!__all_sync(0xffffffffu, mb_wait(&full[slot], par))) {
                            ok = false;
                            if ((tid & 31) == 0) atomicExch(err, 2);
                            break;
                        }
                        const uint32_t st = ring + (uint32_t)slot * A.sstride;
                        q0[(ph + 2 * R) % QN] = lds128(st + A.off_q + own);
                        q1[(ph + 2 * R) % QN] = lds128(st + A.off_q + own + rowb);
                        const unsigned g = (unsigned)z * plane + gxy;
                        const unsigned g0 = (unsigned)z * plane + (unsigned)(y0 * n1);
                        const float4 m0 = q0[(ph + R) % QN], m1 = q1[(ph + R) % QN];
                        // sums of the two rows' points: (row, x)
                        float2 s00 = make_float2(0.f, 0.f), s01 = s00, s10 = s00, s11 = s00;
                        if (KB) {
                            slabx_kb(st, st + cofs, vown, vrow, g0, A, s00, s01, s10, s11);
                            if (A.nslot > A.nst) {
                                if (st0) slabx_kb_far(st + cofs, g, patom, pval, A, s00, s01);
                                if (st1) slabx_kb_far(st + cofs, g + (unsigned)n1, patom, pval, A, s10, s11);
                            }
                        }
                        const uint32_t T = st + (uint32_t)(R + ty) * rowb;
                        slabx_x(T, xc, A, m0, s00, s01);
                        slabx_x(T + rowb, xc, A, m1, s10, s11);
                        // y: each halo row is read once for both rows
                        s00 = fma2v(A.cy[1], lo2(m1), s00);
                        s01 = fma2v(A.cy[1], hi2(m1), s01);
                        s10 = fma2v(A.cy[1], lo2(m0), s10);
                        s11 = fma2v(A.cy[1], hi2(m0), s11);
                        uint32_t Tu = T + (uint32_t)gx * 8u, Td = Tu + rowb;
#pragma unroll
                        for (int r = 1; r <= R; ++r) {
                            Tu -= rowb;
                            Td += rowb;
                            const float4 up = lds128(Tu), dn = lds128(Td);
                            s00 = fma2v(A.cy[r], lo2(up), s00);
                            s01 = fma2v(A.cy[r], hi2(up), s01);
                            s10 = fma2v(A.cy[r], lo2(dn), s10);
                            s11 = fma2v(A.cy[r], hi2(dn), s11);
                            if (r < R) {
                                s00 = fma2v(A.cy[r + 1 <= R ? r + 1 : R], lo2(dn), s00);
                                s01 = fma2v(A.cy[r + 1 <= R ? r + 1 : R], hi2(dn), s01);
                                s10 = fma2v(A.cy[r + 1 <= R ? r + 1 : R], lo2(up), s10);
                                s11 = fma2v(A.cy[r + 1 <= R ? r + 1 : R], hi2(up), s11);
                            }
                        }
#pragma unroll
                        for (int r = 1; r <= R; ++r) {
                            const float4 u0 = q0[(ph + R + r) % QN], d0 = q0[(ph + R - r + QN) % QN];
                            const float4 u1 = q1[(ph + R + r) % QN], d1 = q1[(ph + R - r + QN) % QN];
                            s00 = fma2v(A.cz[r], add2(lo2(u0), lo2(d0)), s00);
                            s01 = fma2v(A.cz[r], add2(hi2(u0), hi2(d0)), s01);
                            s10 = fma2v(A.cz[r], add2(lo2(u1), lo2(d1)), s10);
                            s11 = fma2v(A.cz[r], add2(hi2(u1), hi2(d1)), s11);
                        }
                        {   // the diagonal, by far the largest term, comes last: a sum is rounded to what it already holds
                            const uint32_t va = st + A.off_v + ((g0 + A.vmis) & 3u) * 4u + vown;
                            const float2 v0 = lds64(va), v1 = lds64(va + vrow);
                            s00 = fma2(A.c0 + v0.x, lo2(m0), s00);
                            s01 = fma2(A.c0 + v0.y, hi2(m0), s01);
                            s10 = fma2(A.c0 + v1.x, lo2(m1), s10);
                            s11 = fma2(A.c0 + v1.y, hi2(m1), s11);
                        }
                        float2 t00 = make_float2(0.f, 0.f), t01 = t00, t10 = t00, t11 = t00;
                        if (PREV) {
                            const float4 p0 = lds128(st + A.off_prev + own), p1 = lds128(st + A.off_prev + own + rowb);
                            t00 = mul2(A.mbeta, lo2(p0));
                            t01 = mul2(A.mbeta, hi2(p0));
                            t10 = mul2(A.mbeta, lo2(p1));
                            t11 = mul2(A.mbeta, hi2(p1));
                        }
                        s00 = fma2v(A.alpha, s00, t00);
                        s01 = fma2v(A.alpha, s01, t01);
                        s10 = fma2v(A.alpha, s10, t10);
                        s11 = fma2v(A.alpha, s11, t11);
                        if (st0) *reinterpret_cast<float4*>(Zg + g) = make_float4(s00.x, s00.y, s01.x, s01.y);
                        if (st1) *reinterpret_cast<float4*>(Zg + g + n1) = make_float4(s10.x, s10.y, s11.x, s11.y);
                        // this warp has read the stage: release it to the producer
                        __syncwarp();
                        if ((tid & 31) == 0) mb_arrive(&empty[slot]);
                        if (++slot == D) {
                            slot = 0;
                            par ^= 1u;
                        }
                    }
                }
            }
            f += z1 - z0;
        }
    }
    // every thread reaches this barrier; then drain the copies the producer issued so that none is in flight when the
    // CTA's shared memory is released
    __syncthreads();
    if (tid == ncomp) {
        for (int j = max(0, issued - D); j < issued; ++j)
            if (!mb_wait(&full[j % D], (j / D) & 1)) break;
    }
}

struct SlabxShape {
    int ty = 0, nslab = 0, nthreads = 0, depth = 0, nst = 0;
    unsigned off_q, off_prev, off_v, off_ka, off_kv, off_c, kbytes, sstride;
    size_t smem = 0;
};

// rows per CTA: as many as the threads hold, evened out over the slabs; up to four KB slots staged, fewer where the
// ring would not keep three stages
SlabxShape slabx_shape(const sdft_ctx* c, int nslot) {
    SlabxShape s;
    const int n1 = c->n[0], n2 = c->n[1], hx = n1 / 2;
    const int most = 2 * (SX_COMP / std::max(1, hx));
    if (most < 2) return s;
    s.nslab = (n2 + most - 1) / most;
    s.ty = ((n2 + s.nslab - 1) / s.nslab + 1) / 2 * 2;
    s.nslab = (n2 + s.ty - 1) / s.ty;
    s.nthreads = (hx * (s.ty / 2) + 31) / 32 * 32 + 32;
    const unsigned rowb = n1 * 8u;
    s.kbytes = ((unsigned)(s.ty * n1) * 4u + 8u + 15u) / 16u * 16u;
    for (s.nst = std::min(nslot, 4);; --s.nst) {
        s.off_q = (s.ty + 2 * R) * rowb;
        s.off_prev = s.off_q + s.ty * rowb;
        s.off_v = s.off_prev + s.ty * rowb;
        s.off_ka = s.off_v + s.kbytes;
        s.off_kv = s.off_ka + s.nst * s.kbytes;
        s.off_c = s.off_kv + s.nst * s.kbytes;
        s.sstride = (s.off_c + (unsigned)(c->natom + 2) * 8u + 127u) / 128u * 128u;
        s.depth = (int)std::min<size_t>(SX_MAXD, SX_RING / s.sstride);
        if (s.depth >= 3 || s.nst <= 1) break;
    }
    s.smem = (size_t)s.sstride * s.depth + SX_TAIL;
    return s;
}

}  // namespace

// even n1 (16-byte rows), room for three stages, offsets within a column in 32 bits, real blocks
bool slabx_ok(const sdft_ctx* c, int ncolE) {
    if (c->n[0] % 2 || c->n[0] < 2 * R + 2 || c->n[2] < R || c->opt.boundary != SDFT_BC_PERIODIC || ncolE <= 0) return false;
    int S = 0;
    for (const KBTables& kb : c->kb) {
        if (kb.cplx) return false;
        S = std::max(S, kb.S);
    }
    const SlabxShape s = slabx_shape(c, S);
    return s.ty >= 2 && s.depth >= 3 && c->ng < (1LL << 31) && (long long)ncolE * c->n[2] < (1LL << 30);
}

bool slabx_safe(const sdft_ctx* c, int ncolE) {
    if (!slabx_ok(c, ncolE)) return false;
    int S = 0;
    for (const KBTables& kb : c->kb) S = std::max(S, kb.S);
    const SlabxShape s = slabx_shape(c, S);
    return S <= std::max(4, s.nst + 1) && s.ty >= 8 && c->n[1] >= 2 * R && c->n[2] >= 2 * R;
}

void launch_slabx(sdft_ctx* c, int kpt, const float2* Y, const float2* Yprev, float2* Ynext, int ncolE, const float* V,
                  const float2* kbC, double alpha, double beta, double shift, bool kin, bool timed) {
    SDFT_REQUIRE(kin && V != nullptr, SDFT_ERR_INVALID_ARG, "slab stencil tile needs V and the kinetic term");
    SDFT_REQUIRE(slabx_ok(c, ncolE), SDFT_ERR_INVALID_ARG, "slab stencil tile does not fit");
    SDFT_REQUIRE((((uintptr_t)Y | (uintptr_t)Yprev | (uintptr_t)Ynext) & 15) == 0 && ((uintptr_t)V & 7) == 0,
                 SDFT_ERR_INVALID_ARG, "slab stencil tile: misaligned block");
    const KBTables& kb = c->kb[kpt];
    const bool prev = Yprev != nullptr, haskb = kbC != nullptr && kb.S > 0;
    // the coefficient window of the last group reads at most ncolE * natom + 1 float2 of C
    SDFT_REQUIRE(!haskb || ((kbC == reinterpret_cast<const float2*>(c->C32) ||
                             kbC == reinterpret_cast<const float2*>(c->C32b)) &&
                            (long long)ncolE * c->natom + 1 <= c->c32_elems),
                 SDFT_ERR_INVALID_ARG, "slab stencil tile: KB coefficient buffer too short");
    const SlabxShape s = slabx_shape(c, kb.S);
    SlabxArgs A;
    for (int r = 0; r <= R; ++r) {
        A.cx[r] = make_float2((float)c->coef.cx[r], (float)c->coef.cx[r]);
        A.cy[r] = make_float2((float)c->coef.cy[r], (float)c->coef.cy[r]);
        A.cz[r] = make_float2((float)c->coef.cz[r], (float)c->coef.cz[r]);
    }
    A.c0 = (float)(c->coef.c0 - shift);
    A.alpha = make_float2((float)alpha, (float)alpha);
    A.mbeta = make_float2((float)-beta, (float)-beta);
    A.n1 = c->n[0];
    A.n2 = c->n[1];
    A.n3 = c->n[2];
    A.ty = s.ty;
    A.nslab = s.nslab;
    A.ncolE = ncolE;
    A.natom = c->natom;
    A.nslot = kb.S;
    A.nst = s.nst;
    A.depth = s.depth;
    A.off_q = s.off_q;
    A.off_prev = s.off_prev;
    A.off_v = s.off_v;
    A.off_ka = s.off_ka;
    A.off_kv = s.off_kv;
    A.off_c = s.off_c;
    A.kbytes = s.kbytes;
    A.sstride = s.sstride;
    A.ng = c->ng;
    A.ngl = (unsigned)c->ng;
    A.vmis = (unsigned)((uintptr_t)V >> 2) & 3u;
    // every slab gets the same number of CTAs, which take equal runs of its (pair group, plane) units in the same
    // order (see launch_slab_variant)
    A.total = ncolE * c->n[2];
    const int nper = std::max(1, std::min(sm_count() / s.nslab, A.total));
    A.per_cta = (A.total + nper - 1) / nper;
    ScopedTimer timer(timed ? c : nullptr, SDFT_K_STENCIL,
                      (double)ncolE * (double)c->ng * sizeof(float2) * (prev ? 3.0 : 2.0));
    auto launch = [&](auto kfn) {
        allow_dynamic_smem(kfn, SX_RING + SX_TAIL);
        kfn<<<nper * s.nslab, s.nthreads, s.smem, c->stream>>>(Y, Yprev, Ynext, V, kbC, kb.patom, kb.pval32, A,
                                                               stencil_error_flag(c));
    };
    if (prev && haskb) launch(cheb_slabx_kernel<true, true>);
    else if (!prev && haskb) launch(cheb_slabx_kernel<false, true>);
    else if (prev) launch(cheb_slabx_kernel<true, false>);
    else launch(cheb_slabx_kernel<false, false>);
    SDFT_CUDA(cudaGetLastError());
    count_launch(c);
}

}  // namespace sdft
