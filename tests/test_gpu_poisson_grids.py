"""Mixed-precision Poisson on grids that the multigrid hierarchy does not halve exactly: odd in every dimension, odd after
one halving, mixed parities, and one that coarsens that way twice.  Against the exact Fourier solve, with the bounds of
test_poisson_mixed_multigrid_matches_exact_solve: 1e-9 of the potential at a residual of 1e-11, and at least four times
fewer iterations than the Jacobi scaling needs."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

import workloads  # noqa: E402
from oracle import ham, model  # noqa: E402


@pytest.fixture(scope="module")
def sd():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2005_10431_gb300 import build
    build.build()
    import paper_2005_10431_gb300 as m
    return m


@pytest.mark.parametrize("n", [(27, 27, 27), (29, 40, 31), (54, 54, 54), (47, 26, 50), (46, 50, 46), (61, 63, 107)])
def test_poisson_on_grids_that_do_not_halve(sd, n, monkeypatch):
    cell = workloads.two_atom_cell()
    h = cell.L[0] / cell.n[0]
    cell.n = n
    cell.L = tuple(h * k for k in n)
    f = model.sad_density(cell) + model.pseudocharge(cell)
    ref = ham.poisson_exact(cell, f)
    its = {}
    for mg in ("1", "0"):
        monkeypatch.setenv("SDFT_AAR_MG", mg)
        ctx = sd.sdft_create(cell.L, cell.n, cell.pos, cell.types, cell.species, dict(nstates=8, precision=sd.SDFT_MIXED))
        ft = torch.from_numpy(f).cuda()
        phi = torch.zeros_like(ft)
        its[mg] = sd.sdft_poisson(ctx, ft, phi, 1e-11, 4000)
        assert its[mg] > 0
        assert np.max(np.abs(phi.cpu().numpy() - ref)) < 1e-9 * np.max(np.abs(ref))
        sd.sdft_destroy(ctx)
    assert 4 * its["1"] < its["0"], its
