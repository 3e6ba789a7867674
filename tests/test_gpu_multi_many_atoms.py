"""A multi-cell filter with a cell of so many atoms that its KB coefficients fit beside the column tile but not beside the
brick of the shared launch: every cell is filtered as on its own (FP32, the same sums in the same order in every tile)."""
import dataclasses

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

import workloads  # noqa: E402


@pytest.fixture(scope="module")
def sd():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2005_10431_gb300 import build
    build.build()
    import paper_2005_10431_gb300 as m
    return m


# the wide tile of the 6 x 252 plane takes 74 KB, the coefficients of 20 000 atoms 156 KB of the 227 KB
@pytest.mark.parametrize("natom", [6000, 20000])
def test_cells_of_many_atoms(sd, natom):
    big = workloads.small_cell(npts=8, L=4.0, natom=natom, seed=1, nstates=2)
    big.n, big.L = (6, 252, 8), (31.0, 60.0, 31.0)
    big.pos = np.random.default_rng(6).uniform(0, 1, (natom, 3)) * np.array(big.L)
    big.species = [dataclasses.replace(big.species[0], Z=1e-4, r_loc=0.3, sad_width=0.3, r_cut_proj=1.5)]
    cells = [workloads.small_cell(npts=12, L=4.0, natom=2, seed=2, nstates=8), big,
             workloads.small_cell(npts=14, L=4.0, natom=3, seed=3, nstates=10)]
    ctxs, xs, ys = [], [], []
    for i, c in enumerate(cells):
        ctxs.append(sd.sdft_create(c.L, c.n, c.pos, c.types, c.species, dict(nstates=c.nstates, precision=sd.SDFT_MIXED)))
        sd.sdft_set_veff(ctxs[i], 0, np.random.default_rng(i).normal(0, 0.3, c.ngrid))
        xs.append(sd.pack_block(workloads.initial_orbitals(i, c.ngrid, c.nstates), sd.SDFT_MIXED))
        ys.append(torch.full_like(xs[i], 7.0))
    bounds = [3.0, 3.1, 3.2], [90.0, 160.0, 92.0], [-1.0, -1.1, -1.2]
    sd.sdft_chebyshev_filter_multi(ctxs, xs, ys, 6, *bounds)
    for i, c in enumerate(cells):
        y = torch.empty_like(xs[i])
        sd.sdft_chebyshev_filter(ctxs[i], 0, 0, sd.SDFT_MIXED, xs[i], y, c.nstates, 6, *(b[i] for b in bounds))
        assert torch.equal(ys[i], y)
    with pytest.raises(sd.SdftError) as e:   # refused before anything is launched
        sd.sdft_chebyshev_filter_multi(ctxs, xs, ys, 6, bounds[0], bounds[1], [-1.0, 5.0, -1.2])
    assert e.value.code == -1
    for c in ctxs:
        sd.sdft_destroy(c)
