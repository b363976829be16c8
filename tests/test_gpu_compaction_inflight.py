"""ccr_compact_valid with many requests (the offsets of a request are summed from counts that other blocks turn into offsets meanwhile),
and with several calls of one store in flight: direct ones on one stream, replays of captured ones on another."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

N_DOCS = 10_000


def _batch(rng, n_req, mean):
    lengths = rng.integers(0, 2 * mean + 1, size=n_req)
    lengths[rng.random(n_req) < 0.2] = 0
    lengths[rng.integers(0, n_req)] = 20_001  # several slices
    offsets = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int64)
    idx = rng.integers(-N_DOCS // 2, N_DOCS + 3, size=int(offsets[-1])).astype(np.int32)
    keep = (idx >= 0) & (idx < N_DOCS)
    want = idx[keep], np.concatenate([[0], np.cumsum(keep)])[offsets].astype(np.int64), np.flatnonzero(keep).astype(np.int32)
    return offsets, idx, want


class _Call:
    def __init__(self, store, offsets, idx, want):
        self.store, self.want, self.n_req = store, want, len(offsets) - 1
        self.offsets, self.idx = torch.from_numpy(offsets).cuda(), torch.from_numpy(idx).cuda()
        self.out = torch.full((len(idx) + 1,), -7, dtype=torch.int32, device="cuda")
        self.src = torch.full((len(idx) + 1,), -7, dtype=torch.int32, device="cuda")
        self.offs = torch.full((self.n_req + 2,), -7, dtype=torch.int64, device="cuda")

    def __call__(self, stream=None):
        from paper_2609_22441_b200 import binding as B

        B.ccr_compact_valid(self.store, self.n_req, len(self.idx), self.idx, self.offsets, self.out, self.offs, self.src, stream)

    def check(self):
        kept, offs, src = self.want
        got = self.offs.cpu().numpy()
        assert np.array_equal(got[:-1], offs) and got[-1] == -7
        for have, want in ((self.out, kept), (self.src, src)):
            have = have.cpu().numpy()
            assert np.array_equal(have[:len(want)], want) and (have[len(want):] == -7).all()


@pytest.fixture
def store():
    from paper_2609_22441_b200 import binding as B

    s = B.Docstore(N_DOCS, 8, "float16", 8, "float16")
    yield s
    s.free()


@pytest.mark.parametrize("n_req,mean", [(1, 50), (2, 9_000), (63, 300), (1_022, 40), (1_023, 40), (1_024, 40), (1_025, 40), (2_049, 20), (70_001, 5)])
def test_offsets_of_many_requests(store, n_req, mean):
    call = _Call(store, *_batch(np.random.default_rng(n_req), n_req, mean))
    for _ in range(3):
        call()
    torch.cuda.synchronize()
    call.check()


def test_direct_calls_beside_replays_of_captured_ones(store):
    rng = np.random.default_rng(3)
    captured = [_Call(store, *_batch(rng, n, 200)) for n in (37, 300, 1_500)]
    direct = [_Call(store, *_batch(rng, n, 200)) for n in (41, 290, 1_400, 5)]
    side, graphs = torch.cuda.Stream(), []
    for c in captured:
        c()
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            c()
        graphs.append(g)
    torch.cuda.synchronize()
    for c in captured + direct:
        c.out.fill_(-7), c.src.fill_(-7), c.offs.fill_(-7)
    torch.cuda.synchronize()
    for i in range(150):  # more than 64 calls, so that every word the store could hand out comes round twice
        with torch.cuda.stream(side):
            graphs[i % 3].replay()
        direct[i % 4]()
    torch.cuda.synchronize()
    for c in captured + direct:
        c.check()
    del graphs
