"""Projector tables of atoms whose boxes have very long edges: below and above the length up to which an axis'
displacements are tabulated, and longer than any table that fits in shared memory.  H X (FP64) against the oracle, 1e-12 of
the largest value as in test_gpu_kernels.py: the projector part is some 1e-8 of it, so a wrong or missing
support point shows; its own size is checked against the oracle's as well."""
import dataclasses

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


# edge of the atom's box along x: about 2 (3.3 / L1) n1 points; the other two have 6 or 7
@pytest.mark.parametrize("n1,L1", [(1024, 1.12), (1024, 1.08), (4096, 0.9)])
def test_long_boxes(sd, n1, L1):
    cell = workloads.small_cell(npts=8, L=4.0, natom=2, seed=2, nstates=8)
    cell.n, cell.L = (n1, 6, 6), (L1, 6.0, 6.2)
    cell.pos = np.array([[0.3, 1.1, 2.0], [0.7, 4.3, 5.1]])
    cell.species = [dataclasses.replace(cell.species[0], r_cut_proj=3.3)]
    ctx = sd.sdft_create(cell.L, cell.n, cell.pos, cell.types, cell.species, dict(nstates=8, precision=sd.SDFT_FP64))
    P, E = model.projectors(cell), model.kb_energies(cell)
    # constant along x but for a little: the kinetic part is small, the projections large
    rng = np.random.default_rng(8)
    X = np.repeat(rng.uniform(0.5, 1.5, (2, 36)), n1, axis=1) + 1e-9 * rng.uniform(0, 1, (2, cell.ngrid))
    V = rng.normal(0, 0.3, cell.ngrid)
    sd.sdft_set_veff(ctx, 0, V)
    x = sd.pack_block(X, sd.SDFT_FP64)
    y = torch.empty_like(x)
    sd.sdft_apply_h(ctx, 0, 0, sd.SDFT_FP64, x, y, 2)
    ref = ham.apply_h(cell, X, V, P, E)
    scale = np.max(np.abs(X)) * 0.5 * 3.0 / (L1 / n1) ** 2   # of the terms of the kinetic sum
    err = np.max(np.abs(y.cpu().numpy() - ref))
    assert err < 1e-12 * scale
    kb = np.max(np.abs(ref - ham.apply_h(cell, X, V, 0.0 * P, E)))
    assert kb > 100.0 * 1e-12 * scale   # a projection off by a percent would fail above
    sd.sdft_destroy(ctx)
