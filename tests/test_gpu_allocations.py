"""What a context asks of its allocator: nothing for the descriptors of a learned start beyond the scratch that
sdft_mlp_predict documents; nothing more for moved atoms than the projector tables take; and
tables of a multi-cell filter that do not pile up as cells and degrees grow."""
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


class Counter:
    """The binding's allocator with its calls counted and the live blocks listed."""

    def __init__(self, sd, monkeypatch):
        self.asked, self.live, self._keep = [], {}, []
        make = sd._torch_allocator

        def counted(*args):
            af, ff = make(*args)
            self._keep += [af, ff]

            def alloc(nbytes, user):
                p = af(nbytes, user)
                self.asked.append(nbytes)
                self.live[p] = nbytes
                return p

            def free(p, user):
                self.live.pop(p)
                ff(p, user)

            return type(af)(alloc), type(ff)(free)

        monkeypatch.setattr(sd, "_torch_allocator", counted)


def _ctx(sd, n, natom, precision):
    cell = workloads.small_cell(npts=n, L=0.3 * n, natom=natom, seed=n, nstates=2 * natom + 4)
    return cell, sd.sdft_create(cell.L, cell.n, cell.pos, cell.types, cell.species,
                                dict(nstates=cell.nstates, precision=precision))


def test_descriptors_allocate_nothing(sd, monkeypatch):
    count = Counter(sd, monkeypatch)
    cell, ctx = _ctx(sd, 14, 3, sd.SDFT_FP64)
    feat = torch.empty((cell.ngrid, sd.SDFT_MLP_NFEAT), dtype=torch.bfloat16, device="cuda")
    before = len(count.asked)
    sd.sdft_mlp_dataset(ctx, feat)
    first = feat.clone()
    sd.sdft_mlp_dataset(ctx, feat)
    assert count.asked[before:] == []
    assert torch.equal(feat, first)
    params = torch.tensor(workloads.mlp_init_params(3), device="cuda")
    for _ in range(2):
        sd.sdft_mlp_predict(ctx, params)
    assert count.asked[before:] == [68 * cell.ngrid]   # its documented scratch, once
    sd.sdft_destroy(ctx)
    assert not count.live


def test_moves_keep_the_number_of_blocks(sd, monkeypatch):
    count = Counter(sd, monkeypatch)
    cell, ctx = _ctx(sd, 14, 3, sd.SDFT_FP64)
    blocks, asked = sorted(count.live.values()), []
    for _ in range(3):
        before = len(count.asked)
        sd.sdft_move_atoms(ctx, cell.pos, 0)
        asked.append(len(count.asked) - before)
        assert sorted(count.live.values()) == blocks
    # the projector tables (six by atom, four by point) and their three scratch blocks
    assert asked == [13, 13, 13]
    sd.sdft_destroy(ctx)


def test_tables_of_growing_filters_are_replaced(sd, monkeypatch):
    count = Counter(sd, monkeypatch)
    cells, ctxs, xs = [], [], []
    for i in range(4):
        cell, ctx = _ctx(sd, 12, 2, sd.SDFT_MIXED)
        sd.sdft_set_veff(ctx, 0, torch.zeros(cell.ngrid, dtype=torch.float64, device="cuda"))
        cells.append(cell)
        ctxs.append(ctx)
        xs.append(sd.pack_block(workloads.initial_orbitals(i, cell.ngrid, cell.nstates), sd.SDFT_MIXED))
    ys = [torch.empty_like(x) for x in xs]
    before = len(count.live)
    for n, degree in ((1, 2), (2, 3), (4, 5), (4, 9), (2, 30), (3, 4)):
        sd.sdft_chebyshev_filter_multi(ctxs[:n], xs[:n], ys[:n], degree, [3.0] * n, [90.0] * n, [-1.0] * n)
        assert len(count.live) == before + 2   # the projections' problems and the steps' scalars
    for ctx in ctxs:
        sd.sdft_destroy(ctx)
    assert not count.live


@pytest.mark.parametrize("current", [False, True])
def test_blocks_belong_to_the_contexts_stream(sd, monkeypatch, current):
    # a block released while the context's kernels run must not reach another stream's work
    make, streams = torch.cuda.caching_allocator_alloc, []

    def seen(size, device=None, stream=None):
        streams.append(torch.cuda.current_stream().cuda_stream if stream is None else getattr(stream, "cuda_stream", stream))
        return make(size, device, stream)

    monkeypatch.setattr(torch.cuda, "caching_allocator_alloc", seen)
    own = torch.cuda.Stream()
    cell = workloads.small_cell(npts=12, L=4.0, natom=2, seed=3, nstates=8)
    with torch.cuda.stream(own if current else torch.cuda.default_stream()):
        ctx = sd.sdft_create(cell.L, cell.n, cell.pos, cell.types, cell.species, dict(nstates=8, precision=sd.SDFT_FP64),
                             stream=None if current else own)
    created = len(streams)
    sd.sdft_move_atoms(ctx, cell.pos, 0)   # under the default stream in either case
    assert len(streams) > created > 0
    assert set(streams) == {own.cuda_stream}
    sd.sdft_destroy(ctx)
