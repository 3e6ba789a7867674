"""Descriptors against 64-bit sums over the whole range of BF16, subnormal values included.

Tolerance, in units of the last BF16 place (2^-7 of the power of two below, 2^-133 under 2^-126): 1/2 for the rounding, and
0.01 for what comes before it.  A Gaussian's exponent (down to -87 before the value is subnormal) carries four roundings
of 2^-24 and a constant's 2.1e-8 twice, 2.5e-5 of the value; the power of two, the cut-off function and up to a hundred
additions 7e-6; together 3.2e-5, of a place that is at least 2^-8 of the value: 0.0082."""
import itertools
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

import workloads  # noqa: E402

RC = 6.5


@pytest.fixture(scope="module")
def sd():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2005_10431_gb300 import build
    build.build()
    import paper_2005_10431_gb300 as m
    return m


def _sums(cell):
    axes = [np.arange(cell.n[d]) * cell.h[d] for d in range(3)]
    Z, Y, X = np.meshgrid(axes[2], axes[1], axes[0], indexing="ij")
    X, Y, Z = X.ravel(), Y.ravel(), Z.ravel()
    mu, eta = 6.0 * np.arange(32) / 31.0, 6.0 / 31.0
    G = np.zeros((cell.ngrid, 32))
    reach = [math.ceil(RC / L) + 1 for L in cell.L]
    for p in cell.pos:
        for t in itertools.product(*(range(-k, k + 1) for k in reach)):
            c = p + np.array(t) * np.array(cell.L)
            r = np.sqrt((X - c[0]) ** 2 + (Y - c[1]) ** 2 + (Z - c[2]) ** 2)
            i = np.nonzero(r <= RC)[0]
            if i.size:
                fc = np.sin(np.pi * (RC - r[i]) / (2 * RC)) ** 2
                G[i] += np.exp(-((r[i, None] - mu) ** 2) / (2 * eta * eta)) * fc[:, None]
    return G


@pytest.mark.parametrize("n,L,natom", [((24, 24, 24), (6.0, 6.0, 6.0), 2), ((40, 18, 15), (19.0, 9.0, 8.0), 1),
                                       ((9, 21, 14), (2.5, 7.0, 4.0), 1)])
def test_descriptors_round_64_bit_sums(sd, n, L, natom):
    cell = workloads.small_cell(npts=8, L=4.0, natom=natom, seed=3)
    cell.n, cell.L = n, L
    cell.pos = np.random.default_rng(natom).uniform(0, 1, (natom, 3)) * np.array(L)
    ctx = sd.sdft_create(cell.L, cell.n, cell.pos, cell.types, cell.species,
                         dict(nstates=2 * natom + 4, precision=sd.SDFT_FP64))
    feat = torch.empty((cell.ngrid, sd.SDFT_MLP_NFEAT), dtype=torch.bfloat16, device="cuda")
    sd.sdft_mlp_dataset(ctx, feat)
    got, ref = feat.cpu().double().numpy(), _sums(cell)
    place = 2.0 ** (np.floor(np.log2(np.maximum(ref, 2.0 ** -126))) - 7)
    assert np.max(np.abs(got - ref) / place) <= 0.51
    assert np.sum((ref > 0) & (ref < 2.0 ** -126)) > 0 or natom > 1   # subnormal values were among them
    sd.sdft_destroy(ctx)
