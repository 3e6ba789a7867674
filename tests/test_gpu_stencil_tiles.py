"""Brick stencil tiles against the oracle at the sizes where they can go wrong: ragged tiles and z chunks,
tiles that span the periodic edge, pieces shorter than the stencil, several KB slots per point, odd grids, Bloch
phases, one column and many.

Tolerances as in test_gpu_kernels.py: FP32 H X 2e-5 of the largest value, a degree-m filter 3e-5 m; FP64 1e-12
and 1e-11."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

import workloads  # noqa: E402
from oracle import chefsi, ham, model  # noqa: E402

BRICK8, BRICK4 = (16, "brick8"), (17, "brick4")
SLABX = (18, "slabx")
CBRICK8, CBRICK4 = (5, "brick8"), (6, "brick4")


@pytest.fixture(scope="module")
def sd():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2005_10431_gb300 import build
    build.build()
    import paper_2005_10431_gb300 as m
    return m


def _cell(n, natom):
    """atoms clustered in a corner of the cell, so that up to all of their projector spheres overlap at a point and
    some cross the periodic edges."""
    c = workloads.small_cell(npts=8, L=4.0, natom=natom, seed=21, nstates=2 * natom + 4)
    c.n, c.L = n, tuple(0.3 * k for k in n)
    c.pos = np.random.default_rng(5).uniform(-1.5, 2.5, (natom, 3)) + np.array([0.0, 0.0, 0.5])
    return c


def _check(sd, cell, precision, ns, variant, kred, degree, monkeypatch):
    cplx = any(kred)
    if variant is not None:
        monkeypatch.setenv("SDFT_STENCIL_VARIANT", str(variant[0]))
    ctx = sd.sdft_create(cell.L, cell.n, cell.pos, cell.types, cell.species,
                         dict(nstates=max(ns, cell.nstates), precision=precision), kpts=[kred] if cplx else None)
    V = np.random.default_rng(17).normal(0, 0.4, cell.ngrid)
    sd.sdft_set_veff(ctx, 0, V)
    X = workloads.initial_orbitals(19, cell.ngrid, ns, complex_valued=cplx)
    x = sd.pack_block(X, precision)
    y = torch.full_like(x, 7.0)
    P, E = model.projectors(cell, kred), model.kb_energies(cell)
    err = lambda ref: np.max(np.abs(sd.unpack_block(y, precision, cplx) - ref)) / np.max(np.abs(ref))  # noqa: E731
    sd.sdft_apply_h(ctx, 0, 0, precision, x, y, ns)
    assert err(ham.apply_h(cell, X, V, P, E, kred)) < (2e-5 if precision else 1e-12)
    if variant is not None:
        assert sd.sdft_get_stencil_variant(ctx, cplx) == variant
    sd.sdft_chebyshev_filter(ctx, 0, 0, precision, x, y, ns, degree, 3.0, 90.0, -1.5)
    ref = chefsi.chebyshev_filter(lambda Z: ham.apply_h(cell, Z, V, P, E, kred), X, degree, 3.0, 90.0, -1.5)
    assert err(ref) < (3e-5 * degree if precision else 1e-11)


@pytest.mark.parametrize("n,ns,natom", [((6, 7, 6), 2, 1), ((9, 10, 11), 6, 3), ((37, 11, 9), 4, 4), ((65, 8, 17), 2, 2),
                                        ((8, 70, 6), 10, 5)])
@pytest.mark.parametrize("variant", [BRICK8, BRICK4])
def test_brick_tile_matches_oracle(sd, n, ns, natom, variant, monkeypatch):
    _check(sd, _cell(n, natom), sd.SDFT_MIXED, ns, variant, (0.0, 0.0, 0.0), 3, monkeypatch)


# rows in one slab and in several, a ragged last slab of one row, halos that wrap more than once, an odd number of
# points per plane pair (copies that start between 16-byte boundaries), more KB slots than are staged, odd numbers of pairs
@pytest.mark.parametrize("n,ns,natom", [((14, 7, 6), 2, 1), ((14, 9, 15), 6, 7), ((82, 15, 9), 4, 4), ((46, 27, 13), 10, 2),
                                        ((160, 9, 7), 6, 3), ((22, 30, 40), 14, 5)])
def test_slab_of_any_even_row_matches_oracle(sd, n, ns, natom, monkeypatch):
    _check(sd, _cell(n, natom), sd.SDFT_MIXED, ns, SLABX, (0.0, 0.0, 0.0), 3, monkeypatch)


@pytest.mark.parametrize("n,ns,natom", [((6, 7, 6), 2, 1), ((23, 12, 9), 3, 4), ((7, 37, 13), 5, 2)])
@pytest.mark.parametrize("variant", [CBRICK8, CBRICK4])
def test_complex_brick_tile_matches_oracle(sd, n, ns, natom, variant, monkeypatch):
    _check(sd, _cell(n, natom), sd.SDFT_MIXED, ns, variant, (0.25, -0.375, 0.5), 3, monkeypatch)


@pytest.mark.parametrize("n,ns,kred", [((6, 7, 6), 1, (0, 0, 0)), ((37, 9, 11), 3, (0, 0, 0)), ((13, 24, 9), 9, (0, 0, 0)),
                                       ((7, 19, 10), 3, (0.5, 0.25, -0.125))])
def test_fp64_brick_matches_oracle(sd, n, ns, kred, monkeypatch):
    _check(sd, _cell(n, 3), sd.SDFT_FP64, ns, None, kred, 3, monkeypatch)
