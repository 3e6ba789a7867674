// Instantiations of the fused stencil / Chebyshev-step kernels (see stencil_impl.cuh)
// for FP32 blocks (two lanes per element: an orbital pair, or re/im of a Bloch orbital).
#include "stencil_brick.cuh"

#include <vector>

namespace sdft {
namespace {
// variants timed by the autotuner.  Column tiles: (TX, TY, queue prefetch PF, min blocks per SM,
// cp.async stages D).  Row tiles: (TY rows of full x extent, PF, min blocks per SM, D).
template <int TY, int MAXT, int D>
bool row_ok(const sdft_ctx* c, int ncolE) { return row_variant_ok<TY, MAXT, D>(c, ncolE); }

// row variants: (CPLX, TY, PF, max threads, min blocks per SM, D)
const StepVariant<float2> kReal[] = {
    {&launch_variant<float2, false, 32, 8, 2, 2, 4>, nullptr, "col32x8"},
    {&launch_variant<float2, false, 32, 8, 3, 2, 3>, nullptr, "col32x8pf3"},
    {&launch_variant<float2, false, 32, 16, 2, 1, 3>, nullptr, "col32x16"},
    {&launch_variant<float2, false, 32, 4, 2, 4, 4>, nullptr, "col32x4"},
    {&launch_variant<float2, false, 32, 8, 2, 3, 3>, nullptr, "col32x8occ3"},
    {&launch_variant<float2, false, 32, 8, 2, 4, 3>, nullptr, "col32x8occ4"},
    {&launch_variant<float2, false, 32, 4, 2, 6, 3>, nullptr, "col32x4occ6"},
    {&launch_row_variant<false, 4, 1, 256, 2, 3>, &row_ok<4, 256, 3>, "row4", &launch_row_group<false, 4, 1, 256, 2, 3>},
    {&launch_row_variant<false, 8, 1, 512, 1, 3>, &row_ok<8, 512, 3>, "row8", &launch_row_group<false, 8, 1, 512, 1, 3>},
    {&launch_row_variant<false, 5, 2, 320, 1, 3>, &row_ok<5, 320, 3>, "row5", &launch_row_group<false, 5, 2, 320, 1, 3>},
    {&launch_row_variant<false, 6, 2, 384, 1, 3>, &row_ok<6, 384, 3>, "row6", &launch_row_group<false, 6, 2, 384, 1, 3>},
    // TMA-fed slab tiles (stencil_tma.cu): (n1, TY rows, NP pairs, RY rows per thread, KB slots, stages,
    // min blocks per SM)
    {&launch_slab_variant<80, 8, 2, 1, 2, 3, 1>, &slab_variant_ok<80, 8, 2, 2, 3>, "slab80"},
    {&launch_slab_variant<80, 8, 1, 1, 2, 4, 1>, &slab_variant_ok<80, 8, 1, 2, 4>, "slab80np1"},
    {&launch_slab_variant<120, 8, 1, 1, 2, 4, 1>, &slab_variant_ok<120, 8, 1, 2, 4>, "slab120"},
    {&launch_slab_variant<40, 8, 2, 1, 2, 4, 1>, &slab_variant_ok<40, 8, 2, 2, 4>, "slab40"},
    {&launch_slab_variant<80, 8, 1, 2, 2, 4, 1>, &slab_variant_ok<80, 8, 1, 2, 4>, "slab80ry2"},
    // bricks of 8 and 4 planes (stencil_brick.cuh)
    {&launch_brick<float2, false, 8, 2>, &brick_ok<float2, 8>, "brick8"},
    {&launch_brick<float2, false, 4, 2>, &brick_ok<float2, 4>, "brick4"},
    {&launch_slabx, &slabx_ok, "slabx"},
};
const StepVariant<float2> kCplx[] = {
    {&launch_variant<float2, true, 32, 8, 2, 2, 4>, nullptr, "col32x8"},
    {&launch_variant<float2, true, 32, 8, 3, 2, 3>, nullptr, "col32x8pf3"},
    {&launch_row_variant<true, 4, 1, 256, 2, 3>, &row_ok<4, 256, 3>, "row4", &launch_row_group<true, 4, 1, 256, 2, 3>},
    {&launch_row_variant<true, 8, 1, 256, 2, 3>, &row_ok<8, 256, 3>, "row8", &launch_row_group<true, 8, 1, 256, 2, 3>},
    {&launch_row_variant<true, 10, 1, 256, 2, 3>, &row_ok<10, 256, 3>, "row10", &launch_row_group<true, 10, 1, 256, 2, 3>},
    {&launch_brick<float2, true, 8, 2>, &brick_ok<float2, 8>, "brick8"},
    {&launch_brick<float2, true, 4, 2>, &brick_ok<float2, 4>, "brick4"},
};
constexpr int kRealBrick8 = 16, kCplxBrick8 = 5;   // the brick4 variants follow
constexpr int kRealSlabx = 18;
constexpr unsigned long long kSlabs = 0x1fULL << 11 | 1ULL << kRealSlabx;   // the TMA-fed slab tiles of kReal
constexpr int kNReal = sizeof(kReal) / sizeof(kReal[0]);
constexpr int kNCplx = sizeof(kCplx) / sizeof(kCplx[0]);
}  // namespace

// Real blocks with rows of 44 points and more (even) for which slabx_safe() holds: only the slab tiles are timed.  us a
// step, slab and best column, row or brick tile: 80^3, 180 columns 294 and 668; 82 x 82 x 76, 176 columns 358 and 706;
// 96^3, 300 columns 915 and 1600; 64 x 60 x 60, 66 columns 63 and 115; 48^3, 32 columns 23 and 27; 160 x 40 x 40, 60
// columns (4 slots) 119 and 132.  Shorter rows: 40^3 20.7 and 21.9, 36^3 19.0 and 18.9, 20^3 27 and 18.  Where it does not
// hold: KB slots past the staged ones (four at most) are read from L2 by few threads, 64 x 60 x 60, 80 columns with 5, 9,
// 21 slots 132 and 153, 221 and 175, 501 and 238; 80^3, 140 columns with 6, 52 slots 650 and 538, 4290 and 990; slabs of
// 6, 4, 2 rows re-read their halo, 200 x 40 x 40 157 and 150, 256 x 40 x 40 218 and 205, 400 x 30 x 30 294 and 175; thin
// axes do too, 60 x 7 x 400 160 and 121.
static bool long_rows(const sdft_ctx* c, bool cplx, int ncolE) { return !cplx && c->n[0] >= 44 && slabx_safe(c, ncolE); }

// Cells whose projectors overlap so much that the column tile is ahead of the bricks, which read the KB slots with few
// warps: more than seven slots at a point on average, and a block that fills the GPU with column tiles.  us a step, column
// tile and brick of 8 planes at 6, 8, 12 slots: 40^3, 20 columns 51 and 45, 59 and 62, 57 and 81; 10 columns 45 and 27, 53
// and 37, 50 and 47; Bloch, 60 x 50 x 50, 20 columns 155 and 157, 190 and 196, 243 and 291; 40^3, 20 columns 108 and
// 74, 121 and 100, 130 and 129.
static bool dense_kb(const sdft_ctx* c, bool cplx, int ncolE) {
    double mean = 0.0;
    for (const KBTables& kb : c->kb) mean = std::max(mean, kb.mean);
    return mean > 7.0 && (double)c->ng * ncolE > (cplx ? 2.5e6 : 5e5);
}

// Calls too small to be timed take a brick tile: 37 x 41 x 45 points, 20 columns: 15.4 us a step, 31 with the column
// tile; 40^3, 28 columns: 20 and 26; 48^3, 40 columns: 35 and 66.  Bricks of 8 planes need two CTAs an SM, else 4.
// (The slab would take 29 us for the last of these, but the multi-cell filter runs bricks, and a cell gets the same bits
// from it as from its own filter.)
static int small_variant(const sdft_ctx* c, bool cplx, int ncolE) {
    const int v8 = cplx ? kCplxBrick8 : kRealBrick8;
    if (!brick_ok<float2, 8>(c, ncolE) || dense_kb(c, cplx, ncolE)) return 0;
    const BrickTile t = brick_tile(c->n[0], c->n[1]);
    const long long ctas8 = (long long)t.tiles_x * t.tiles_y * ((c->n[2] + 7) / 8) * ncolE;
    return ctas8 >= 2 * 152 ? v8 : v8 + 1;
}

template <>
void launch_kb_project<float2>(sdft_ctx* c, int kpt, const float2* Y, float2* C, int ncolE) {
    launch_project_impl<float2>(c, kpt, Y, C, ncolE);
}

template <>
void launch_cheb_step<float2>(sdft_ctx* c, int kpt, const float2* Y, const float2* Yprev, float2* Ynext, int ncolE,
                              const float* V, const float2* kbC, double alpha, double beta, double shift,
                              bool with_kinetic) {
    const bool cplx = c->kb[kpt].cplx;
    const StepVariant<float2>* table = cplx ? kCplx : kReal;
    const int nvar = cplx ? kNCplx : kNReal;
    int& choice = c->stencil_choice[cplx ? 1 : 0];
    int pick = choice;
    // the row and slab tiles move 16-byte vectors: blocks that start in between take a brick
    const bool aligned = (((uintptr_t)Y | (uintptr_t)Yprev | (uintptr_t)Ynext) & 15) == 0;
    if (!aligned) {
        pick = small_variant(c, cplx, ncolE);
    } else if (pick < 0) {
        // when the caller wants the output's KB coefficients too, the variants are timed with them (fused
        // or by the separate pass, into the caller's target buffer, which the real launch then rewrites)
        float2* kb_next = c->kb_next;
        c->kb_next = nullptr;
        bool fused = true;
        pick = autotune_stencil<float2>(c, table, nvar, kpt, Y, Yprev, Ynext, ncolE, V, kbC, alpha, beta, shift,
                                        kb_next, kb_next ? &launch_kb_project<float2> : nullptr, &fused,
                                        long_rows(c, cplx, ncolE) ? kSlabs : ~0ULL);
        c->kb_next = kb_next;
        if (pick >= 0) {   // small calls are not timed and do not fix the choice
            choice = pick;
            if (kb_next) c->stencil_fuse = fused;
        } else {
            pick = small_variant(c, cplx, ncolE);
        }
    }
    if (!c->stencil_fuse) c->kb_next = nullptr;   // the separate projection pass was timed faster
    c->kb_next_done = false;
    // the chosen variant may not fit this call (another column count): fall back to the column tile
    const int v = (table[pick].ok == nullptr || table[pick].ok(c, ncolE)) ? pick : 0;
    c->stencil_last[cplx ? 1 : 0] = v;
    c->stencil_last_name[cplx ? 1 : 0] = table[v].name;
    table[v].fn(c, kpt, Y, Yprev, Ynext, ncolE, V, kbC, alpha, beta, shift, with_kinetic, true);
}

// scalar FP32, Laplacian-only: the correction solves of the mixed-precision Poisson solver
template <>
void launch_cheb_step<float>(sdft_ctx* c, int kpt, const float* Y, const float* Yprev, float* Ynext, int ncolE,
                             const float* V, const float* kbC, double alpha, double beta, double shift,
                             bool with_kinetic) {
    launch_variant<float, false, 32, 8, 2, 2, 3>(c, kpt, Y, Yprev, Ynext, ncolE, V, kbC, alpha, beta, shift,
                                                 with_kinetic, true);
}


// grouped FP32 launches: the row variant used is the autotuned one when it is a row tile that
// fits, else the first row tile that fits; -1 if none does (callers then loop over problems)
int group_variant_f32(sdft_ctx* c, bool cplx, int ncolE) {
    const StepVariant<float2>* table = cplx ? kCplx : kReal;
    const int nvar = cplx ? kNCplx : kNReal;
    const int ch = c->stencil_choice[cplx ? 1 : 0];
    if (ch >= 0 && table[ch].group && table[ch].ok(c, ncolE)) return ch;
    for (int v = 0; v < nvar; ++v)
        if (table[v].group && table[v].ok(c, ncolE)) return v;
    return -1;
}

// time every fitting row variant on one grouped launch (tab: a table whose Ynext may be
// overwritten) and return the fastest
int autotune_group_f32(sdft_ctx* c, bool cplx, const RowProblem* grp, int nprob, int ncolE, bool haskb) {
    const StepVariant<float2>* table = cplx ? kCplx : kReal;
    const int nvar = cplx ? kNCplx : kNReal;
    if (const char* env = getenv("SDFT_STENCIL_VARIANT")) {
        const int v = atoi(env);
        if (v >= 0 && v < nvar && table[v].group && table[v].ok(c, ncolE)) return v;
    }
    cudaEvent_t a, b;
    SDFT_CUDA(cudaEventCreate(&a));
    SDFT_CUDA(cudaEventCreate(&b));
    int best = -1;
    float best_ms = 1e30f;
    for (int v = 0; v < nvar; ++v) {
        if (!table[v].group || !table[v].ok(c, ncolE)) continue;
        table[v].group(c, 0, grp, nprob, ncolE, false, haskb);   // warm-up
        SDFT_CUDA(cudaEventRecord(a, c->stream));
        for (int r = 0; r < 2; ++r) table[v].group(c, 0, grp, nprob, ncolE, false, haskb);
        SDFT_CUDA(cudaEventRecord(b, c->stream));
        SDFT_CUDA(cudaEventSynchronize(b));
        float ms = 0.f;
        SDFT_CUDA(cudaEventElapsedTime(&ms, a, b));
        if (ms < best_ms) {
            best_ms = ms;
            best = v;
        }
    }
    cudaEventDestroy(a);
    cudaEventDestroy(b);
    return best;
}

void launch_group_step_f32(sdft_ctx* c, bool cplx, int variant, const RowProblem* grp, int nprob, int ncolE,
                           bool prev, bool haskb) {
    const StepVariant<float2>* table = cplx ? kCplx : kReal;
    c->stencil_last[cplx ? 1 : 0] = variant;
    c->stencil_last_name[cplx ? 1 : 0] = table[variant].name;
    table[variant].group(c, 0, grp, nprob, ncolE, prev, haskb);
}

// ---- several cells in one launch (independent grids, FP32 real blocks) --------------------
// One cell of a multi-cell filter.  The table is written once per filter call: the blocks of step k follow from
// the ring buffers and k, and the recurrence scalars of every (step, cell) come from a device table.
struct MultiProblem {
    StepArgs<float> A;                // grid, coefficients, shift
    const float2* X;                  // the filter's input
    float2* ring[3];                  // step k writes ring[slot(k)], see multi_slot
    const float* V;
    const float2* C;
    const int* patom;
    const void* pval;
    int nslot, tw, th, tiles_x, cta_begin, cta_end;
};
__host__ __device__ inline int multi_slot(int k, int m) { return (((2 - (m - k)) % 3) + 3) % 3; }
constexpr int MULTI_ZC = 8;
__constant__ MultiProblem c_multi[MULTI_MAX];

// step k of degree m; grid: the CTAs of every cell, cell p owning [cta_begin, cta_end) = tiles x z chunks x columns
template <bool PREV>
__global__ void __launch_bounds__(BRICK_NT, 2) brick_multi_kernel(const int nprob, const int k, const int m,
                                                                 const float2* __restrict__ steps) {
    const int b = blockIdx.x;
    int lo = 0, hi = nprob - 1;       // the cell whose range holds b
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (b < c_multi[mid].cta_end) hi = mid;
        else lo = mid + 1;
    }
    const MultiProblem& P = c_multi[lo];
    int local = b - P.cta_begin;
    const int tiles = P.tiles_x * ((P.A.n2 + P.th - 1) / P.th);
    const int tile = local % tiles;
    local /= tiles;
    const int zc = local % P.A.nzc, col = local / P.A.nzc;
    const int by = tile / P.tiles_x, bx = tile - by * P.tiles_x;
    const float2* Y = k == 1 ? P.X : P.ring[multi_slot(k - 1, m)];
    const float2* Yprev = k == 1 ? nullptr : (k == 2 ? P.X : P.ring[multi_slot(k - 2, m)]);
    const float2 ab = steps[(long long)(k - 1) * nprob + lo];
    brick_body<float2, false, MULTI_ZC, PREV, true>(Y, Yprev, P.ring[multi_slot(k, m)], P.V, P.C, P.patom, P.pval,
                                                    P.nslot, P.A, ab.x, ab.y, P.tw, P.th, bx, by, zc * MULTI_ZC, col);
}

void chebyshev_filter_multi(const std::vector<sdft_ctx*>& ctxs, const std::vector<const void*>& X,
                            const std::vector<void*>& Y, int m, const double* a, const double* b, const double* a0) {
    const int n = (int)ctxs.size();
    SDFT_REQUIRE(m >= 1, SDFT_ERR_INVALID_ARG, "degree must be >= 1");
    SDFT_REQUIRE(n >= 1 && n <= MULTI_MAX, SDFT_ERR_INVALID_ARG, "multi-cell launch takes 1..64 cells");
    for (int i = 0; i < n; ++i)
        SDFT_REQUIRE(b[i] > a[i] && a[i] > a0[i], SDFT_ERR_INVALID_ARG, "filter bounds must satisfy a0 < a < b");
    // cells whose KB coefficients do not fit beside a brick (some 5000 atoms and more), or that fill the GPU and take
    // another tile (dense_kb), are filtered on their own
    std::vector<int> fit;
    for (int i = 0; i < n; ++i)
        if (brick_ok<float2, MULTI_ZC>(ctxs[i], ctxs[i]->nfilt / 2) && !dense_kb(ctxs[i], false, ctxs[i]->nfilt / 2))
            fit.push_back(i);
    if ((int)fit.size() < n) {
        std::vector<sdft_ctx*> cs;
        std::vector<const void*> xs;
        std::vector<void*> ys;
        std::vector<double> as, bs, a0s;
        for (int i = 0, q = 0; i < n; ++i) {
            if (q < (int)fit.size() && fit[q] == i) {
                ++q;
                cs.push_back(ctxs[i]);
                xs.push_back(X[i]);
                ys.push_back(Y[i]);
                as.push_back(a[i]);
                bs.push_back(b[i]);
                a0s.push_back(a0[i]);
            } else {
                sdft_ctx* c = ctxs[i];
                chebyshev_filter(c, 0, SDFT_MIXED, X[i], Y[i], c->nfilt, m, a[i], b[i], a0[i], c->veff, c->veff32);
            }
        }
        if (!cs.empty()) chebyshev_filter_multi(cs, xs, ys, m, as.data(), bs.data(), a0s.data());
        return;
    }
    sdft_ctx* c0 = ctxs[0];
    // per cell: grid, tile, ring of its own block buffers (T1, T2, Y), recurrence scalars of every step
    std::vector<MultiProblem> probs(n);
    std::vector<float2> steps((size_t)m * n);
    long long total = 0;
    size_t dsm = 0;
    double elems = 0;
    for (int i = 0; i < n; ++i) {
        sdft_ctx* c = ctxs[i];
        const double e = 0.5 * (b[i] - a[i]), cc = 0.5 * (b[i] + a[i]);
        const double sigma1 = e / (a0[i] - cc);
        double sigma = sigma1;
        for (int k = 1; k <= m; ++k) {
            double alpha = sigma1 / e, beta = 0.0;
            if (k > 1) {
                const double s2 = 1.0 / (2.0 / sigma1 - sigma);
                alpha = 2.0 * s2 / e;
                beta = sigma * s2;
                sigma = s2;
            }
            steps[(size_t)(k - 1) * n + i] = make_float2((float)alpha, (float)beta);
        }
        MultiProblem& P = probs[i];
        const int nzc = (c->n[2] + MULTI_ZC - 1) / MULTI_ZC;
        P.A = make_args<float>(c, 0, 0.0, 0.0, cc, MULTI_ZC, nzc);
        P.X = (const float2*)X[i];
        int got = 0;
        for (int k = 0; k < 4 && got < 2; ++k)
            if (c->blk[k] != X[i] && c->blk[k] != Y[i]) P.ring[got++] = (float2*)c->blk[k];
        SDFT_REQUIRE(got == 2, SDFT_ERR_INVALID_ARG, "no free block buffers for the filter");
        P.ring[2] = (float2*)Y[i];
        P.V = c->veff32;
        P.C = (const float2*)c->C32;
        P.patom = c->kb[0].patom;
        P.pval = c->kb[0].pval32;
        P.nslot = c->kb[0].S;
        const BrickTile t = brick_tile(c->n[0], c->n[1]);
        P.tw = t.tw;
        P.th = t.th;
        P.tiles_x = t.tiles_x;
        P.cta_begin = (int)total;
        total += (long long)t.tiles_x * t.tiles_y * nzc * (c->nfilt / 2);
        SDFT_REQUIRE(total < (1LL << 31), SDFT_ERR_INVALID_ARG, "multi-cell launch too large");
        P.cta_end = (int)total;
        dsm = std::max(dsm, brick_smem<float2>(t, MULTI_ZC, c->natom));
        elems += (double)(c->nfilt / 2) * (double)c->ng;
    }
    // KB projections of every (step, cell): one table, uploaded once, one grouped launch per step
    std::vector<KBProblem> ktab;
    std::vector<int> kcell;
    int max_natom = 0, max_ncolE = 0;
    for (int i = 0; i < n; ++i) {
        const KBTables& kb = ctxs[i]->kb[0];
        if (kb.S == 0 || kb.natom == 0) continue;
        kcell.push_back(i);
        max_natom = std::max(max_natom, kb.natom);
        max_ncolE = std::max(max_ncolE, ctxs[i]->nfilt / 2);
    }
    const int nk = (int)kcell.size();
    ktab.reserve((size_t)m * nk);
    for (int k = 1; k <= m; ++k)
        for (int i : kcell) {
            sdft_ctx* c = ctxs[i];
            const KBTables& kb = c->kb[0];
            const float2* cur = k == 1 ? probs[i].X : probs[i].ring[multi_slot(k - 1, m)];
            ktab.push_back(KBProblem{cur, c->C32, kb.cnt, kb.idx, kb.val32, kb.gamma, kb.cap, kb.natom, c->nfilt / 2,
                                     c->ng});
        }
    // the tables grow with degree and cells; an outgrown one is given back once nothing reads it any more
    auto grow = [&](auto*& table, int& cap, int need) {
        if (cap >= need) return;
        if (table) {
            SDFT_CUDA(cudaStreamSynchronize(c0->stream));
            ctx_release(c0, table);
            table = nullptr;
            cap = 0;
        }
        table = reinterpret_cast<std::remove_reference_t<decltype(table)>>(ctx_alloc(c0, sizeof(*table) * (size_t)need));
        cap = need;
    };
    grow(c0->m_ktab, c0->m_ktab_cap, (int)ktab.size());
    grow(c0->m_steps, c0->m_steps_cap, m * n);
    // pageable sources: the copies are staged before the calls return, so the vectors may go out of scope
    if (nk > 0)
        SDFT_CUDA(cudaMemcpyAsync(c0->m_ktab, ktab.data(), sizeof(KBProblem) * ktab.size(), cudaMemcpyHostToDevice,
                                  c0->stream));
    SDFT_CUDA(cudaMemcpyAsync(c0->m_steps, steps.data(), sizeof(float2) * steps.size(), cudaMemcpyHostToDevice,
                              c0->stream));
    SDFT_CUDA(cudaMemcpyToSymbolAsync(c_multi, probs.data(), sizeof(MultiProblem) * n, 0, cudaMemcpyHostToDevice,
                                      c0->stream));
    auto step = [&](auto kfn, int k) {
        ScopedTimer timer(c0, SDFT_K_STENCIL, elems * sizeof(float2) * (k > 1 ? 3.0 : 2.0));
        if (dsm > 48 * 1024) allow_dynamic_smem(kfn, BRICK_SMEM_MAX);
        kfn<<<(unsigned)total, BRICK_NT, dsm, c0->stream>>>(n, k, m, c0->m_steps);
        SDFT_CUDA(cudaGetLastError());
        count_launch(c0);
    };
    for (int k = 1; k <= m; ++k) {
        if (nk > 0)
            launch_group_project_f32(c0, false, c0->m_ktab + (size_t)(k - 1) * nk, nk, max_natom, max_ncolE);
        if (k > 1) step(brick_multi_kernel<true>, k);
        else step(brick_multi_kernel<false>, k);
    }
}

void launch_group_project_f32(sdft_ctx* c, bool cplx, const KBProblem* grp, int nprob, int natom, int ncolE) {
    launch_project<float2>(c, nullptr, nullptr, nullptr, natom, ncolE, nprob, cplx, grp);
}

}  // namespace sdft
