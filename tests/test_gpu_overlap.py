"""Joins launched back to back on one stream may overlap on the device; whatever they leave must be what one after the
other would leave.  Batches of different sizes are joined alternately into the SAME output buffers, with a padded join
that has nothing to store in between, and the last state is compared byte for byte with the CPU oracle."""
import numpy as np
import pytest

from oracle import oracle
from paper_2609_22441_b200 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("second", [False, True])
@pytest.mark.parametrize("n_req,big,small", [(1, 60_000, 40), (3, 20_000, 500), (8, 30_000, 33)])  # the last: one of each kernel
def test_alternating_batches_into_one_buffer(n_req, big, small, second):
    from paper_2609_22441_b200 import binding as B

    wls = [W.config1(seed=5 + i, n_docs=200_000, n_req=n_req, n_cand=n, second_degree=second, edge_lo=40, edge_hi=3_000) for i, n in enumerate((big, small))]
    wls[1].store = wls[0].store
    wants = [oracle.join_workload(wl, n_threads=4) for wl in wls]
    store = B.store_from_workload(wls[0])
    dbs = [B.DeviceBatch(wl.batch) for wl in wls]
    out_b = store.out_row_bytes(0)
    rows = torch.zeros((dbs[0].total_cands, out_b), dtype=torch.uint8, device="cuda")
    mask = torch.zeros(dbs[0].total_cands, dtype=torch.uint8, device="cuda")
    # compacted offsets that keep nothing: the padded join over them stores no row of its own
    none_kept = torch.zeros(n_req + 1, dtype=torch.int64, device="cuda")
    T, M = (torch.zeros(s, dtype=torch.uint8, device="cuda") for s in ((n_req, 1, out_b), (n_req, 1)))

    def join(db):
        B.ccr_join_batch(store, db.n_req, db.total_cands, db.max_edge_len, db.edge_keys, db.edge_feats, db.edge_offsets, db.cand_idx,
                         db.cand_offsets, db.req_feats, rows, mask)

    def nothing(db):
        B.ccr_join_batch_padded(store, db.n_req, db.total_cands, db.max_edge_len, 1, db.edge_keys, db.edge_feats, db.edge_offsets, db.cand_idx,
                                none_kept, db.req_feats, T, M)

    torch.cuda.synchronize()
    for _ in range(30):
        join(dbs[0])
        nothing(dbs[1])
        join(dbs[1])
        join(dbs[0])
        join(dbs[1])
    torch.cuda.synchronize()
    got_rows, got_mask, n = rows.cpu().numpy(), mask.cpu().numpy(), dbs[1].total_cands
    assert np.array_equal(got_mask[:n], wants[1][1]) and np.array_equal(got_rows[:n], wants[1][0])
    assert np.array_equal(got_mask[n:], wants[0][1][n:]) and np.array_equal(got_rows[n:], wants[0][0][n:])
    assert not T.any() and store.device_status() == B.CCR_OK
    store.free()


@pytest.mark.parametrize("second", [False, True])
@pytest.mark.parametrize("front_ws", [False, True])
def test_small_join_reads_what_the_join_in_front_wrote(second, front_ws):
    """A small join is in stream order with everything in front of it, its inputs included: its candidate positions are the rows
    of the join launched directly before it.  Two such joins write the buffer in turn, so an early read would find the other's."""
    from paper_2609_22441_b200 import binding as B

    rng = np.random.default_rng(17)
    back = W.config1(seed=31, n_docs=50_000, n_req=1, n_cand=64, second_degree=second, edge_lo=900, edge_hi=900)
    fronts = []
    for i in range(2):  # rows of 64 bytes of positions and a 16-byte edge section
        st = W.make_store(rng, 5_000, 25_000, 16, np.float32)
        st.doc_feats = rng.integers(0, back.store.n_docs, size=(st.n_docs, 16)).astype(np.int32).view(np.float32)
        keys, _ = W.make_viewer(rng, 25_000, 1_000, 8, np.float16)
        feats = rng.integers(0, 40, size=(1_000, 8)).astype(np.uint16).view(np.float16)
        cands = rng.integers(0, st.n_docs, size=6_000).astype(np.int32)
        fronts.append(W.Workload("front", i, st, W.assemble_batch([keys], [feats], [cands], None, 8, np.float16, 0, np.float32)))
    wants = []
    for wl in fronts:
        idx = np.ascontiguousarray(oracle.join_workload(wl, n_threads=4)[0]).view(np.int32).reshape(-1)
        b = back.batch
        b2 = W.assemble_batch([b.edge_keys], [b.edge_feats], [idx], b.req_feats, b.edge_dim, b.edge_dtype, b.req_dim, b.req_dtype)
        wants.append(oracle.join_workload(W.Workload("back", 0, back.store, b2), n_threads=4))
    n = fronts[0].batch.total_cands * 20
    front_stores, dbs = [B.store_from_workload(wl) for wl in fronts], [B.DeviceBatch(wl.batch) for wl in fronts]
    store, db = B.store_from_workload(back), B.DeviceBatch(back.batch)
    idx_buf = torch.zeros(n, dtype=torch.int32, device="cuda")
    front_mask = torch.zeros(n // 20, dtype=torch.uint8, device="cuda")
    co = torch.tensor([0, n], dtype=torch.int64, device="cuda")
    outs = [(torch.zeros((n, store.out_row_bytes(0)), dtype=torch.uint8, device="cuda"), torch.zeros(n, dtype=torch.uint8, device="cuda")) for _ in range(2)]
    flags = B.CCR_FLAG_WARP_SPECIALISED if front_ws else 0
    torch.cuda.synchronize()
    for _ in range(20):
        for st, d, (rows, mask) in zip(front_stores, dbs, outs):
            B.ccr_join_batch(st, 1, d.total_cands, d.max_edge_len, d.edge_keys, d.edge_feats, d.edge_offsets, d.cand_idx, d.cand_offsets, None, idx_buf,
                             front_mask, flags)
            B.ccr_join_batch(store, 1, n, db.max_edge_len, db.edge_keys, db.edge_feats, db.edge_offsets, idx_buf, co, db.req_feats, rows, mask)
    torch.cuda.synchronize()
    for (rows, mask), (want_rows, want_mask) in zip(outs, wants):
        assert np.array_equal(mask.cpu().numpy(), want_mask) and np.array_equal(rows.cpu().numpy(), want_rows)
    for st in front_stores + [store]:
        assert st.device_status() == B.CCR_OK
        st.free()


@pytest.mark.parametrize("k", [28_400, 28_540, 28_700, 28_790])
def test_forced_staging_of_the_longest_lists(k):
    """Lists that just fit the two-phase kernel's shared memory are staged whole, with and without room for anything beside them."""
    from paper_2609_22441_b200 import binding as B

    wl = W.config1(seed=77, n_docs=60_000, n_req=1, n_cand=3_001, edge_lo=k, edge_hi=k)
    assert wl.batch.max_edge_len == k
    want_rows, want_mask = oracle.join_workload(wl, n_threads=4)
    store, db = B.store_from_workload(wl), B.DeviceBatch(wl.batch)
    rows, mask = B.join_batch(store, db, B.CCR_FLAG_FORCE_SMEM)
    torch.cuda.synchronize()
    assert np.array_equal(mask.cpu().numpy(), want_mask) and np.array_equal(rows.cpu().numpy(), want_rows)
    store.free()


@pytest.mark.parametrize("second", [False, True])
def test_positions_written_between_two_joins_on_many_streams_and_in_graphs(second):
    """Joins with a kernel between them that writes the second one's candidate positions, on more streams than a store keeps the last
    join of, launched and captured; the launches of a replay stand beside direct ones on other streams."""
    from paper_2609_22441_b200 import binding as B

    wl = W.config1(seed=3, n_docs=120_000, n_req=6, n_cand=24_000, second_degree=second)
    b = wl.batch
    cand_b = np.random.default_rng(4).permutation(b.cand_idx)
    wants = [oracle.join_workload(w, n_threads=4) for w in (wl, W.Workload("b", 0, wl.store, W.Batch(**{**b.__dict__, "cand_idx": cand_b})))]
    store, db = B.store_from_workload(wl), B.DeviceBatch(b)
    cands = [db.cand_idx, torch.from_numpy(cand_b).cuda()]
    out_b = store.out_row_bytes()
    streams = [torch.cuda.Stream() for _ in range(11)]
    bufs = [dict(scratch=cands[0].clone(), rows=torch.zeros((b.total_cands, out_b), dtype=torch.uint8, device="cuda"),
                 mask=torch.zeros(b.total_cands, dtype=torch.uint8, device="cuda")) for _ in streams]

    def join(buf, idx, st):
        B.ccr_join_batch(store, db.n_req, db.total_cands, db.max_edge_len, db.edge_keys, db.edge_feats, db.edge_offsets, idx, db.cand_offsets,
                         db.req_feats, buf["rows"], buf["mask"], 0, st)

    def steps(i, buf, st):  # ends with batch i % 2 in the rows
        join(buf, cands[1 - i % 2], st)
        buf["scratch"].copy_(cands[i % 2])
        join(buf, buf["scratch"], st)

    torch.cuda.synchronize()
    graphs = []
    for k in range(2):
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=streams[k]):
            steps(k, bufs[k], streams[k])
            steps(k + 1, bufs[k], streams[k])
        graphs.append(g)
    torch.cuda.synchronize()
    for i in range(12):
        for k, st in enumerate(streams):
            with torch.cuda.stream(st):
                if k < len(graphs):
                    graphs[k].replay()
                else:
                    steps(i + k, bufs[k], st)
    torch.cuda.synchronize()
    for k, buf in enumerate(bufs):
        want_rows, want_mask = wants[(k + 1) % 2 if k < len(graphs) else (11 + k) % 2]
        assert np.array_equal(buf["mask"].cpu().numpy(), want_mask) and np.array_equal(buf["rows"].cpu().numpy(), want_rows)
    assert store.device_status() == B.CCR_OK
    store.free()


def test_joins_of_two_stores_in_turn_with_an_upsert_into_one_of_them():
    """The join in front may be another store's.  Rows and ids of the second store change between the joins of a round."""
    from paper_2609_22441_b200 import binding as B

    wls = [W.config1(seed=40 + i, n_docs=60_000, n_req=8, n_cand=20_000) for i in range(2)]
    stores, dbs = [B.store_from_workload(wl) for wl in wls], [B.DeviceBatch(wl.batch) for wl in wls]
    s, b = wls[1].store, wls[1].batch
    rng = np.random.default_rng(2)
    pos = rng.permutation(s.n_docs).astype(np.int32)
    news = [(rng.standard_normal(s.doc_feats.shape).astype(s.doc_feats.dtype), rng.permutation(s.author_ids)) for _ in range(2)]
    wants = []
    for doc, auth in news:
        st = oracle.upsert(s.doc_feats.copy(), s.author_ids.copy(), pos.astype(np.int64), doc, auth)
        wants.append(oracle.join(st[0], st[1], b.edge_keys, b.edge_feats, b.edge_offsets, b.cand_idx, b.cand_offsets, req_feats=b.req_feats, n_threads=4))
    want0 = oracle.join_workload(wls[0], n_threads=4)
    dev = [tuple(torch.from_numpy(a).cuda() for a in (pos, *n)) for n in news]
    outs = [[torch.zeros((db.total_cands, st.out_row_bytes()), dtype=torch.uint8, device="cuda"), torch.zeros(db.total_cands, dtype=torch.uint8, device="cuda")]
            for st, db in ((stores[0], dbs[0]), (stores[1], dbs[1]), (stores[1], dbs[1]))]
    torch.cuda.synchronize()
    for i in range(30):
        B.join_batch(stores[0], dbs[0], 0, *outs[0])
        stores[1].upsert(*dev[i % 2])
        B.join_batch(stores[1], dbs[1], 0, *outs[1 + i % 2])
        B.join_batch(stores[0], dbs[0], 0, *outs[0])
    torch.cuda.synchronize()
    for (rows, mask), (want_rows, want_mask) in zip(outs, [want0] + wants):
        assert np.array_equal(mask.cpu().numpy(), want_mask) and np.array_equal(rows.cpu().numpy(), want_rows)
    for st in stores:
        assert st.device_status() == B.CCR_OK
        st.free()
