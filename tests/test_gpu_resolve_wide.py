"""GPU parity of ccr_resolve_ids at the batch sizes where large batches begin (the level below the top staged in shared memory),
around the index sizes at which a level is added, against the CPU oracle."""
import numpy as np
import pytest

from oracle import oracle

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n_q", [(1 << 18) - 1, 1 << 18, (1 << 20) + 33])
@pytest.mark.parametrize("n_ids", [1, 2_055, 16_383, 16_392, 131_071, 131_135, 1_000_003, 9_000_000])
def test_batches_around_the_wide_top(n_ids, n_q):
    from paper_2609_22441_b200 import binding as B

    rng = np.random.default_rng(n_ids + n_q)
    ids = np.cumsum(rng.integers(1, 4, size=n_ids)) * 2
    pos = rng.permutation(n_ids).astype(np.int32)
    q = ids[rng.integers(0, n_ids, size=n_q)] + (rng.random(n_q) < 0.1)
    q[:4] = [ids[0], ids[-1], ids[0] - 1, ids[-1] + 1]
    index = B.IdIndex(torch.from_numpy(ids).cuda(), torch.from_numpy(pos).cuda())
    got = index.resolve(torch.from_numpy(q).cuda()).cpu().numpy()
    assert np.array_equal(got, oracle.resolve_ids(ids, q, pos))
    index.free()
