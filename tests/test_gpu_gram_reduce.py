"""Split sums of the CUDA-core Gram at numbers of splits and columns that give an element's lanes different trip counts:
one term, a few, one past a multiple of a pass over all lanes (128), two passes and a remainder, and so many columns that
the elements take more than one round of the grid.

Tolerance: each split adds its products in FP32, at most 2 `CHUNK` of them per component (the two parts of a complex
product), so an element is off by at most 2 CHUNK + 2 roundings of 2^-24 of the sum of the products' magnitudes; the
splits are added in FP64."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

CHUNK = 32   # points per split at these sizes (the kernel's granule)


@pytest.fixture(scope="module")
def sd():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2005_10431_gb300 import build
    build.build()
    import paper_2005_10431_gb300 as m
    return m


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("ncol,nsplit", [(2, 1), (20, 7), (20, 9), (20, 127), (20, 129), (20, 137), (20, 259), (290, 11)])
def test_split_sums(sd, ncol, nsplit, cplx):
    ng = CHUNK * nsplit - 5
    rng = np.random.default_rng(100 * ncol + nsplit)
    # all of one sign, so that a lost or doubled partial sum is 1 / nsplit of an element
    Y, HY = rng.uniform(0.5, 1.5, (2, ncol, ng))
    if cplx:
        Y, HY = Y + 1j * rng.uniform(0.5, 1.5, (ncol, ng)), HY + 1j * rng.uniform(0.5, 1.5, (ncol, ng))
    st = np.complex64 if cplx else np.float32
    Y, HY = Y.astype(st), HY.astype(st)
    y, hy = sd.pack_block(Y, sd.SDFT_MIXED), sd.pack_block(HY, sd.SDFT_MIXED)
    shape = (ncol, ncol, 2) if cplx else (ncol, ncol)
    m, hs = (torch.full(shape, 7.0, dtype=torch.float64, device="cuda") for _ in range(2))
    sd.sdft_subspace_matrices_noalloc(sd.SDFT_MIXED, cplx, y, hy, ng, ncol, m, hs)
    Y, HY = Y.astype(np.complex128 if cplx else np.float64), HY.astype(np.complex128 if cplx else np.float64)
    for got, other in ((m, HY * 0 + Y), (hs, HY)):
        a = got.cpu().numpy()
        a = (a[..., 0] + 1j * a[..., 1] if cplx else a).T   # column-major
        upper = np.triu(np.conj(Y) @ other.T)
        ref = upper + np.conj(np.triu(upper, 1).T)
        np.fill_diagonal(ref, np.real(np.diag(ref)))
        size = np.abs(Y) @ np.abs(other).T
        size = np.triu(size) + np.triu(size, 1).T
        assert np.all(np.abs(a - ref) <= (2 * CHUNK + 2) * 2.0 ** -24 * np.sqrt(2.0) * size)
