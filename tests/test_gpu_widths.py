"""GPU parity of the run-time-width row movement, byte for byte against the CPU oracle: rows whose loaded sections make
2 ... 208 sixteen-byte chunks, around one and two batches of loads (20 chunks a lane first-degree, 8 second-degree)
and around whole rows per warp step (16, 32, 64 chunks), with partial groups, misses and unresolved positions."""
import numpy as np
import pytest

from oracle import oracle

from helpers import gpu_join, tiny_workload

pytestmark = pytest.mark.gpu
pytest.importorskip("torch")

# (doc_dim float32, edge_dim float16, req_dim float32) -> doc_dim / 4 + edge_dim / 8 + req_dim / 4 chunks
WIDTHS = ((4, 8, 0), (4, 8, 4), (20, 16, 4), (24, 16, 0), (28, 8, 8), (56, 16, 0), (60, 32, 4), (64, 32, 4), (64, 64, 32), (100, 48, 4),
          (104, 48, 4), (128, 64, 0), (128, 64, 4), (224, 64, 0), (768, 64, 32))


@pytest.mark.parametrize("second", [False, True])
@pytest.mark.parametrize("doc_dim,edge_dim,req_dim", WIDTHS)
def test_every_width_matches_the_oracle(doc_dim, edge_dim, req_dim, second):
    from paper_2609_22441_b200 import binding as B

    wl = tiny_workload(doc_dim + 7 * edge_dim + req_dim, 150, 90, 6, 60, 230, second, req_dim, doc_dim=doc_dim, edge_dim=edge_dim,
                       sum_mask=0xF0F0A5A5F0F0A5A5)
    want_rows, want_mask = oracle.join_workload(wl, n_threads=4)
    store, db = B.store_from_workload(wl), B.DeviceBatch(wl.batch)
    try:
        for flags in (0, B.CCR_FLAG_WARP_SPECIALISED, B.CCR_FLAG_WARP_SPECIALISED | B.CCR_FLAG_NO_REBALANCE):
            rows, mask = gpu_join(store, db, flags)
            assert np.array_equal(mask, want_mask) and np.array_equal(rows, want_rows), flags
    finally:
        store.free()
