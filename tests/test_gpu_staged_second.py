"""GPU parity of the second-degree join whose document rows pass through shared memory: rows of the tuned widths, groups and sub-tiles of
every remainder, groups without any document, the largest bound on the list length that 16-bit match indices hold and the next
one, ragged and padded output."""
import numpy as np
import pytest

from oracle import oracle
from paper_2609_22441_b200 import workloads as W

from helpers import gpu_join, tiny_workload

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _workload(seed, edge_dim, req_dim, lengths):
    wl = tiny_workload(seed, 900, 3_000, len(lengths), 700, 1, True, req_dim, doc_dim=128, doc_dtype=np.float16, edge_dim=edge_dim,
                       sum_mask=0xA5A5_0FF0_3C3C_FFFF & ((1 << edge_dim) - 1))
    rng = np.random.default_rng(seed + 1)
    b = wl.batch
    b.cand_offsets = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int64)
    b.cand_idx = rng.integers(-1, wl.store.n_docs + 1, size=int(b.cand_offsets[-1])).astype(np.int32)
    b.cand_idx[40:140] = -1  # whole groups without a document
    return wl


@pytest.mark.parametrize("edge_dim,req_dim", [(32, 0), (32, 16), (64, 0), (64, 16)])
@pytest.mark.parametrize("bound", [0, 65_534, 65_535])
def test_remainders_bounds_and_empty_groups(edge_dim, req_dim, bound):
    from paper_2609_22441_b200 import binding as B

    lengths = [1, 0, 31, 32, 33, 127, 128, 129, 5_000, 0, 4_095, 255]
    wl = _workload(edge_dim + req_dim, edge_dim, req_dim, lengths)
    want_rows, want_mask = oracle.join_workload(wl)
    store = B.store_from_workload(wl)
    db = B.DeviceBatch(wl.batch)
    db.max_edge_len = max(db.max_edge_len, bound)
    for flags in (B.CCR_FLAG_WARP_SPECIALISED, B.CCR_FLAG_WARP_SPECIALISED | B.CCR_FLAG_FORCE_GLOBAL):
        rows, mask = gpu_join(store, db, flags)
        assert np.array_equal(mask, want_mask) and np.array_equal(rows, want_rows)
    T, M, offs, src = B.join_batch_padded(store, db, n_max=4_097)
    torch.cuda.synchronize()
    s, b = wl.store, wl.batch
    want = oracle.join_padded(s.doc_feats, s.author_ids, b.edge_keys, b.edge_feats, b.edge_offsets, b.cand_idx, b.cand_offsets, n_max=4_097,
                              req_feats=b.req_feats, actor_ids=s.actor_ids, actor_types=s.actor_types, reduce_sum_mask=s.reduce_sum_mask)
    assert np.array_equal(T.cpu().numpy(), want[0]) and np.array_equal(M.cpu().numpy(), want[1])
    assert store.device_status() == B.CCR_OK
    store.free()


def test_back_to_back_and_on_two_streams():
    """Launches that overlap on one stream and run at the same time on two."""
    from paper_2609_22441_b200 import binding as B

    wl = W.config1(n_docs=40_000, n_req=24, n_cand=9_001, second_degree=True)
    want_rows, want_mask = oracle.join_workload(wl, n_threads=4)
    store = B.store_from_workload(wl)
    db = B.DeviceBatch(wl.batch)
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    outs = [(torch.empty((db.total_cands, store.out_row_bytes()), dtype=torch.uint8, device="cuda"),
             torch.empty(db.total_cands, dtype=torch.uint8, device="cuda")) for _ in streams]
    torch.cuda.synchronize()
    for i in range(12):
        B.join_batch(store, db, 0, *outs[i % 2], stream=streams[i % 2])
    torch.cuda.synchronize()
    for rows, mask in outs:
        assert np.array_equal(rows.cpu().numpy(), want_rows) and np.array_equal(mask.cpu().numpy(), want_mask)
    assert store.device_status() == B.CCR_OK
    store.free()


@pytest.mark.parametrize("edge_dim", [32, 64])
def test_rows_and_ids_written_by_the_upsert_in_front(edge_dim):
    """Two batches of documents replace the same rows in turn, each followed by a join without a synchronisation in between."""
    from paper_2609_22441_b200 import binding as B

    n, lengths = 50_000, [9_000] * 20
    wl = _workload(edge_dim, edge_dim, 16, lengths)
    rng = np.random.default_rng(edge_dim)
    s, b = wl.store, wl.batch
    reps = n // s.n_docs + 1
    s.doc_feats, s.author_ids, s.actor_ids, s.actor_types = (np.ascontiguousarray(np.concatenate([a] * reps)[:n])
                                                             for a in (s.doc_feats, s.author_ids, s.actor_ids, s.actor_types))
    s.n_docs = n
    b.cand_idx = rng.integers(0, n, size=b.total_cands).astype(np.int32)
    store, db = B.store_from_workload(wl), B.DeviceBatch(b)
    pos = rng.permutation(n).astype(np.int32)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    batches, wants, outs = [], [], []
    for _ in range(2):
        order = rng.permutation(n)
        new = (rng.standard_normal(s.doc_feats.shape).astype(np.float16), s.author_ids[order], s.actor_ids[order], s.actor_types[order])
        state = oracle.upsert(s.doc_feats.copy(), s.author_ids.copy(), pos.astype(np.int64), new[0], new[1], s.actor_ids.copy(), s.actor_types.copy(),
                              new[2], new[3])
        wants.append(oracle.join(state[0], state[1], b.edge_keys, b.edge_feats, b.edge_offsets, b.cand_idx, b.cand_offsets, req_feats=b.req_feats,
                                 actor_ids=state[2], actor_types=state[3], reduce_sum_mask=s.reduce_sum_mask, n_threads=4))
        batches.append([dev(a) for a in new])
        outs.append((torch.zeros((b.total_cands, store.out_row_bytes()), dtype=torch.uint8, device="cuda"),
                     torch.zeros(b.total_cands, dtype=torch.uint8, device="cuda")))
    pos = dev(pos)
    torch.cuda.synchronize()
    for i in range(20):
        store.upsert(pos, *batches[i % 2])
        B.join_batch(store, db, 0, *outs[i % 2])
    torch.cuda.synchronize()
    for (rows, mask), (want_rows, want_mask) in zip(outs, wants):
        assert np.array_equal(mask.cpu().numpy(), want_mask) and np.array_equal(rows.cpu().numpy(), want_rows)
    assert store.device_status() == B.CCR_OK
    store.free()


@pytest.mark.parametrize("total,max_len", [((1 << 20) - 1, 700), (1 << 20, 700), ((1 << 20) + 77, 700), ((1 << 20) + 77, 5_000), ((1 << 20) + 77, 5_100)])
def test_64_byte_edge_rows_on_both_sides_of_the_rule(total, max_len):
    """Document rows of 64-byte edge rows are staged from 2^20 candidates on, while a list of the promised length fits beside its table."""
    from paper_2609_22441_b200 import binding as B

    lengths = [300_000, 33, 0, 200_001, 31, 1]
    lengths.append(total - sum(lengths))
    wl = _workload(total + max_len, 32, 0, lengths)
    want_rows, want_mask = oracle.join_workload(wl, n_threads=8)
    store, db = B.store_from_workload(wl), B.DeviceBatch(wl.batch)
    db.max_edge_len = max(db.max_edge_len, max_len)
    rows, mask = gpu_join(store, db, 0)
    assert np.array_equal(mask, want_mask) and np.array_equal(rows, want_rows)
    assert store.device_status() == B.CCR_OK
    store.free()
