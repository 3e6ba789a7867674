"""Atom-centred grid fields against the oracle where the row kernels' splits change: several periodic images
per axis, rows longer than a CTA, more (atom, image) candidates than a CTA tests at once, odd sizes.

Tolerances: the fields are sums of products of three FP64 exponentials (a few ulp each, all of one sign), so
1e-12 of the largest value; a BF16 descriptor is its FP32 sum (1e-5 relative at worst, the Gaussians' arguments)
rounded to 8 bits, so 2^-8 relative."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

import workloads  # noqa: E402
from oracle import mlp, model  # noqa: E402


@pytest.fixture(scope="module")
def sd():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2005_10431_gb300 import build
    build.build()
    import paper_2005_10431_gb300 as m
    return m


@pytest.mark.parametrize("n,L,natom", [((9, 10, 11), (3.6, 4.0, 4.4), 3), ((261, 7, 6), (60.0, 5.0, 4.0), 2),
                                       ((6, 33, 8), (7.0, 21.5, 6.1), 5), ((31, 12, 10), (12.0, 6.0, 5.0), 40)])
def test_fields_and_descriptors_match_oracle(sd, n, L, natom):
    cell = workloads.small_cell(npts=8, L=4.0, natom=natom, seed=13, nstates=2 * natom + 4)
    cell.n, cell.L = n, L
    cell.pos = np.random.default_rng(4).uniform(-0.2, 1.2, (natom, 3)) * np.array(L)   # some outside the cell
    ctx = sd.sdft_create(cell.L, cell.n, cell.pos, cell.types, cell.species,
                         dict(nstates=cell.nstates, precision=sd.SDFT_FP64))
    for got, ref in ((sd.sdft_get_pseudocharge(ctx), model.pseudocharge(cell)),
                     (sd.sdft_get_sad_density(ctx), model.sad_density(cell))):
        assert np.max(np.abs(got - ref)) < 1e-12 * np.max(np.abs(ref))
    feat = torch.empty((cell.ngrid, sd.SDFT_MLP_NFEAT), dtype=torch.bfloat16, device="cuda")
    sd.sdft_mlp_dataset(ctx, feat)
    G = feat.float().cpu().numpy().astype(np.float64)
    ref = mlp.descriptors(cell)
    assert np.all(np.abs(G - ref) <= 2.0 ** -8 * np.abs(ref) + 1e-30)
