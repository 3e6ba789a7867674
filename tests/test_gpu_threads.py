"""Contexts on their own host threads and streams: cells whose stencil tiles need different amounts of shared memory (above
the 48 KB that a kernel takes without asking) filter at the same time and give what they give alone."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

import workloads  # noqa: E402

REPEATS = 400


@pytest.fixture(scope="module")
def sd():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2005_10431_gb300 import build
    build.build()
    import paper_2005_10431_gb300 as m
    return m


@pytest.mark.parametrize("cplx,precision", [(False, 1), (True, 1), (True, 0)])
def test_filters_of_two_threads(sd, cplx, precision):
    jobs = []
    for n in (20, 37):   # tiles of 20 x 10 and 19 x 13 points
        cell = workloads.small_cell(npts=n, L=0.3 * n, natom=2, seed=n, nstates=8)
        stream = torch.cuda.Stream()
        ctx = sd.sdft_create(cell.L, cell.n, cell.pos, cell.types, cell.species, dict(nstates=8, precision=precision),
                             kpts=[(0.25, 0.0, -0.125)] if cplx else None, stream=stream)
        sd.sdft_set_veff(ctx, 0, np.random.default_rng(n).normal(0, 0.3, cell.ngrid))
        x = sd.pack_block(workloads.initial_orbitals(n, cell.ngrid, 4, complex_valued=cplx), precision)
        y, ref = torch.empty_like(x), torch.empty_like(x)
        torch.cuda.synchronize()
        sd.sdft_chebyshev_filter(ctx, 0, 0, precision, x, ref, 4, 8, 3.0, 90.0, -1.0)
        jobs.append((ctx, x, y, ref))
    errors = []

    def work(ctx, x, y, _):
        try:
            for _ in range(REPEATS):
                sd.sdft_chebyshev_filter(ctx, 0, 0, precision, x, y, 4, 8, 3.0, 90.0, -1.0)
        except Exception as e:  # noqa: BLE001
            errors.append(e)

    threads = [threading.Thread(target=work, args=j) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for _, _, y, ref in jobs:
        assert torch.equal(y, ref)
