"""Pseudocharge and superposition density of grids of 2^15 points and more, which sum products of per-axis exponentials,
against the oracle: the first size that takes them, rows longer than a CTA, several periodic images per axis, more
(atom, image) candidates than a CTA tests at once, odd sizes, atoms outside the cell, and an isolated cell (no images).

Tolerance: sums of products of three FP64 exponentials (a few ulp each, all of one sign), so 1e-12 of the largest value."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

import workloads  # noqa: E402
from oracle import model  # noqa: E402


@pytest.fixture(scope="module")
def sd():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2005_10431_gb300 import build
    build.build()
    import paper_2005_10431_gb300 as m
    return m


@pytest.mark.parametrize("n,L,natom,boundary", [
    ((32, 32, 32), (8.2, 8.2, 8.2), 2, "periodic"), ((261, 13, 11), (60.0, 5.0, 4.0), 3, "periodic"),
    ((33, 35, 37), (3.1, 12.5, 6.1), 24, "periodic"), ((31, 40, 28), (12.0, 6.0, 5.0), 40, "periodic"),
    ((33, 32, 35), (11.0, 10.6, 11.6), 3, "dirichlet"), ((259, 12, 13), (40.0, 4.0, 4.3), 2, "dirichlet")])
def test_separable_fields_match_oracle(sd, n, L, natom, boundary):
    cell = workloads.small_cell(npts=8, L=4.0, natom=natom, seed=13, nstates=2 * natom + 4)
    cell.n, cell.L, cell.boundary = n, L, boundary
    assert cell.ngrid >= 1 << 15
    lo, hi = (-0.2, 1.2) if boundary == "periodic" else (0.2, 0.8)
    cell.pos = np.random.default_rng(4).uniform(lo, hi, (natom, 3)) * np.array(L)
    ctx = sd.sdft_create(cell.L, cell.n, cell.pos, cell.types, cell.species,
                         dict(nstates=cell.nstates, precision=sd.SDFT_FP64,
                              boundary=sd.SDFT_BC_DIRICHLET if boundary == "dirichlet" else sd.SDFT_BC_PERIODIC))
    for got, ref in ((sd.sdft_get_pseudocharge(ctx), model.pseudocharge(cell)),
                     (sd.sdft_get_sad_density(ctx), model.sad_density(cell))):
        assert np.max(np.abs(got - ref)) < 1e-12 * np.max(np.abs(ref))
    sd.sdft_destroy(ctx)
