"""Small joins (the two-phase kernel): the sampled top of a list that is not staged whole, at the sample counts where a thread's share of
them begins another round, and sub-tiles around what the threads of a block take at a time."""
import numpy as np
import pytest

from oracle import oracle
from paper_2609_22441_b200 import workloads as W

from helpers import gpu_join

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("second", [False, True])
@pytest.mark.parametrize("n_cand,k,sampled", [
    (70, 4_097, False), (342, 5_119, False), (342, 5_120, False), (65, 5_122, False), (300, 10_239, False), (300, 10_244, False), (1_000, 20_481, False),
    (200, 3, True), (200, 5_119, True), (200, 5_120, True), (200, 5_124, True), (200, 10_240, True), (200, 10_245, True),
    (255, 900, False), (1_023, 900, False), (1_024, 900, False), (1_025, 900, False), (75_000, 900, False)])
def test_samples_and_sub_tiles(n_cand, k, sampled, second):
    from paper_2609_22441_b200 import binding as B

    wl = W.config1(seed=n_cand + k, n_docs=30_000 + 2 * n_cand, n_req=1, n_cand=n_cand, edge_lo=k, edge_hi=k, second_degree=second)
    assert wl.batch.max_edge_len == k
    want_rows, want_mask = oracle.join_workload(wl, n_threads=4)
    store, db = B.store_from_workload(wl), B.DeviceBatch(wl.batch)
    for blocks in (0, 1):  # one block per SM: more candidates of a block, several sub-tiles
        store.set_tuning(blocks_per_sm=blocks)
        rows, mask = gpu_join(store, db, B.CCR_FLAG_FORCE_SAMPLED if sampled else 0)
        assert np.array_equal(mask, want_mask) and np.array_equal(rows, want_rows)
    assert store.device_status() == B.CCR_OK
    store.free()
