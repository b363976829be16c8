"""GPU parity of ccr_resolve_ids around the regions of the index (4,096 ids, a hash table each): region edges, ids whose regions span
2^32 and more, queries that share their low 32 bits with an indexed id, and host-sourced indexes that arrive in several chunks."""
import numpy as np
import pytest

from oracle import oracle

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

LOW = 1 << 32


def _ids(rng, n, spread):
    if spread == "dense":
        return np.arange(n, dtype=np.int64) * 3 - 2 * n  # negative ids too
    if spread == "wide":
        return np.unique(rng.integers(-(1 << 62), 1 << 62, size=n + n // 8 + 8))[:n].astype(np.int64)
    gaps = rng.integers(1, 6, size=n)
    gaps[n // 2:n // 2 + 1] += LOW  # one gap of 2^32 somewhere: one region is wide
    return np.cumsum(gaps).astype(np.int64)


@pytest.mark.parametrize("on_device", [False, True])
@pytest.mark.parametrize("spread", ["dense", "wide", "gap"])
@pytest.mark.parametrize("n_ids", [1, 3, 4_095, 4_096, 4_097, 8_192, 8_193, 40_961, 1_000_003])
def test_region_edges_and_shared_low_bits(n_ids, spread, on_device):
    from paper_2609_22441_b200 import binding as B

    rng = np.random.default_rng(n_ids)
    ids = _ids(rng, n_ids, spread)
    assert len(ids) == n_ids
    pos = rng.permutation(n_ids).astype(np.int32) - 7 if n_ids % 2 else None
    edges = ids[np.clip(np.concatenate([np.arange(0, n_ids, 4_096), np.arange(4_095, n_ids, 4_096), [n_ids - 1]]), 0, n_ids - 1)]
    some = ids[rng.integers(0, n_ids, size=3_000)]
    near = np.concatenate([edges, edges - 1, edges + 1, some, some + 1])
    q = np.concatenate([near, near + LOW, near - LOW, near ^ np.int64(LOW), [0, -1, np.iinfo(np.int64).min, np.iinfo(np.int64).max]]).astype(np.int64)
    up = (lambda a: None if a is None else torch.from_numpy(a).cuda()) if on_device else (lambda a: a)
    index = B.IdIndex(up(ids), up(pos))
    got = index.resolve(torch.from_numpy(q).cuda()).cpu().numpy()
    assert np.array_equal(got, oracle.resolve_ids(ids, q, pos))
    index.free()


def test_host_ids_in_several_chunks():
    from paper_2609_22441_b200 import binding as B

    rng = np.random.default_rng(8)
    n = (8 << 20) + 4_097
    ids = np.cumsum(rng.integers(1, 4, size=n)) * 2
    pos = rng.permutation(n).astype(np.int32)
    q = np.concatenate([ids[rng.integers(0, n, size=50_000)] + (rng.random(50_000) < 0.1), ids[(8 << 20) - 5_000:(8 << 20) + 4_097]])
    index = B.IdIndex(ids, pos)
    got = index.resolve(torch.from_numpy(q).cuda()).cpu().numpy()
    assert np.array_equal(got, oracle.resolve_ids(ids, q, pos))
    index.free()
