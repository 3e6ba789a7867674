"""Which FP32 tile a block large enough to be timed gets, where one is far ahead of the others: slab tiles for even rows, but
not for cells with many KB slots at a point (seven times the bricks' time with 20 of them) or with very long rows; and how
many launches a first call spends on the choice."""
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


def _filter(sd, n, natom, spread, ns, calls=1, kred=None, Z=4.0):
    """tile of a filter of `ns` columns, and the launches of each of `calls` calls"""
    cell = workloads.small_cell(npts=8, L=4.0, natom=natom, seed=3, nstates=ns)
    cell.n, cell.L, cell.species = n, tuple(0.2565 * k for k in n), [workloads.Species(Z=Z)]
    cell.pos = np.random.default_rng(natom).uniform(0, spread, (natom, 3)) * np.array(cell.L)
    ctx = sd.sdft_create(cell.L, cell.n, cell.pos, cell.types, cell.species,
                         dict(nstates=ns, precision=sd.SDFT_MIXED, mix_hist=1), kpts=kred)
    sd.sdft_set_veff(ctx, 0, np.random.default_rng(1).normal(0, 0.3, cell.ngrid))
    x = torch.rand((ns if kred else ns // 2, cell.ngrid, 2), device="cuda") - 0.5
    y = torch.empty_like(x)
    launches = []
    for _ in range(calls):
        before = sd.sdft_launch_count(ctx)
        sd.sdft_chebyshev_filter(ctx, 0, 0, sd.SDFT_MIXED, x, y, ns, 3, 3.0, 160.0, -1.5)
        launches.append(sd.sdft_launch_count(ctx) - before)
    name = sd.sdft_get_stencil_variant(ctx, bool(kred))[1]
    sd.sdft_destroy(ctx)
    return name, launches


@pytest.mark.parametrize("n,natom,spread,ns,slab", [
    ((64, 60, 60), 10, 1.0, 80, True),      # up to 4 slots at a point
    ((64, 60, 60), 30, 0.4, 80, False),     # atoms in one corner: 21 slots
    ((60, 50, 50), 100, 1.0, 240, False),   # a dense cell
    ((400, 30, 30), 10, 1.0, 60, False)])   # slabs of two rows
def test_slab_tiles_where_they_are_ahead(sd, n, natom, spread, ns, slab):
    name, _ = _filter(sd, n, natom, spread, ns)
    assert name.startswith("slab") == slab, name


@pytest.mark.parametrize("n,natom,tile", [
    ((40, 40, 40), 8, "brick"), ((40, 40, 40), 110, "col"),   # 0.8 and 11 slots at a point on average
    ((24, 24, 24), 24, "brick")])                             # 12, but too small a block to fill the GPU
def test_untimed_calls(sd, n, natom, tile):
    name, launches = _filter(sd, n, natom, 1.0, 20, calls=2, Z=1.8 * 20 / natom if natom > 8 else 4.0)
    assert name.startswith(tile)
    assert launches[0] == launches[1]


# seven column tiles (Bloch blocks: two) run four times each, with a projection (Bloch: none) after every run, were 56 and 8
# launches; the bricks' tables are longer, and their first calls take no more
@pytest.mark.parametrize("kred,most", [(None, 56), ([(0.25, 0.125, -0.375)], 12)])
def test_first_call_on_odd_rows(sd, kred, most):
    name, launches = _filter(sd, (63, 63, 63), 27, 1.0, 66, calls=2, kred=kred)
    assert name.startswith("brick")
    assert 0 < launches[0] - launches[1] <= most
