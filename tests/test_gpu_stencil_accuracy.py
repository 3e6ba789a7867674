"""Rounding of the FP32 stencil tiles: H X of a tile that replaces the column tile is at least as close to the FP64 result,
in the root mean square over a block (some 1e5 values of random orbitals, so that the figures repeat to a percent)."""
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


@pytest.mark.parametrize("n", [(46, 27, 13), (82, 16, 14)])
@pytest.mark.parametrize("variant", [(16, "brick8"), (18, "slabx")])
def test_tile_rounds_no_worse_than_the_column_tile(sd, n, variant, monkeypatch):
    cell = workloads.small_cell(npts=8, L=4.0, natom=3, seed=21, nstates=10)
    cell.n, cell.L = n, tuple(0.2565 * k for k in n)
    cell.pos = np.random.default_rng(5).uniform(0, 1, (3, 3)) * np.array(cell.L)
    V = np.random.default_rng(17).normal(0, 0.3, cell.ngrid)
    X = workloads.initial_orbitals(19, cell.ngrid, 10).astype(np.float32).astype(np.float64)

    def h_of(precision, tile):
        if tile is not None:
            monkeypatch.setenv("SDFT_STENCIL_VARIANT", str(tile))
        ctx = sd.sdft_create(cell.L, cell.n, cell.pos, cell.types, cell.species, dict(nstates=10, precision=precision))
        sd.sdft_set_veff(ctx, 0, V)
        x = sd.pack_block(X, precision)
        y = torch.empty_like(x)
        sd.sdft_apply_h(ctx, 0, 0, precision, x, y, 10)
        if tile is not None:
            assert sd.sdft_get_stencil_variant(ctx)[0] == tile
        out = sd.unpack_block(y, precision, False)
        sd.sdft_destroy(ctx)
        return out

    exact = h_of(sd.SDFT_FP64, None)
    rms = {t: np.sqrt(np.mean((h_of(sd.SDFT_MIXED, t) - exact) ** 2)) for t in (0, variant[0])}
    assert rms[variant[0]] <= 1.02 * rms[0]
