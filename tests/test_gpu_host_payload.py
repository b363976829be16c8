"""The host-buffer joins with payloads in page-locked, pageable and mixed host memory, aligned and not, with array lengths around
the 16-byte pieces of the transfer kernel, and buffers whose contents change from call to call; byte for byte against the
CPU oracle."""
import numpy as np
import pytest

from oracle import oracle
from paper_2609_22441_b200 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _host(a, how, lead):
    """The array in host memory, `lead` elements behind the start of its allocation."""
    if a is None:
        return None
    flat = torch.from_numpy(np.ascontiguousarray(a).reshape(-1).view(np.uint8))
    step = a.dtype.itemsize
    buf = torch.zeros(flat.numel() + lead * step + 64, dtype=torch.uint8, pin_memory=how == "pinned")
    view = buf[lead * step:lead * step + flat.numel()]
    view.copy_(flat)
    return view


@pytest.mark.parametrize("entry", ["workspace", "static"])
@pytest.mark.parametrize("how,lead", [("pinned", 0), ("pinned", 1), ("pageable", 0), ("mixed", 0)])
@pytest.mark.parametrize("n_req,n_cand,second", [(1, 1, False), (1, 15, True), (2, 17, False), (3, 4097, True), (1, 60_001, False)])
def test_payload_in_any_host_memory(n_req, n_cand, second, how, lead, entry):
    from paper_2609_22441_b200 import binding as B

    wls = [W.config1(seed=40 + i, n_docs=max(3_000, 4 * n_cand), n_req=n_req, n_cand=n_cand, second_degree=second, edge_lo=3, edge_hi=901) for i in range(3)]
    for wl in wls[1:]:
        wl.store = wls[0].store
    store = B.store_from_workload(wls[0])
    out_b = store.out_row_bytes(0)
    most_c, most_e = max(w.batch.total_cands for w in wls), max(int(w.batch.edge_offsets[-1]) for w in wls)
    ws = B.Workspace(store, n_req, most_c, most_e)
    mask = torch.zeros(most_c + 64, dtype=torch.uint8, pin_memory=how != "pageable")[lead:lead + most_c]
    rows = torch.zeros((most_c, out_b), dtype=torch.uint8)
    d_rows, d_mask = torch.zeros((most_c, out_b), dtype=torch.uint8, device="cuda"), torch.zeros(most_c, dtype=torch.uint8, device="cuda")
    names = ("edge_keys", "edge_feats", "edge_offsets", "cand_idx", "cand_offsets", "req_feats")
    kept = {}
    for wl in wls + wls[:1]:
        b = wl.batch
        for i, k in enumerate(names):  # the same buffers again where the lengths allow it, other contents
            new = _host(getattr(b, k), ("pinned", "pageable")[i & 1] if how == "mixed" else how, lead)
            if new is not None and k in kept and kept[k].numel() == new.numel():
                kept[k].copy_(new)
            else:
                kept[k] = new
        args = (b.n_req, b.total_cands, b.max_edge_len, int(b.edge_offsets[-1])) + tuple(kept[k] for k in names)
        want_rows, want_mask = oracle.join_workload(wl, n_threads=4)
        if entry == "workspace":
            B.ccr_join_batch_host(store, ws, *args, rows, mask)
            torch.cuda.synchronize()
            got_rows, got_mask = rows.numpy()[:b.total_cands], mask.numpy()[:b.total_cands]
        else:
            B.ccr_join_payload_static(store, *args, d_rows, d_mask)
            torch.cuda.synchronize()
            got_rows, got_mask = d_rows.cpu().numpy()[:b.total_cands], d_mask.cpu().numpy()[:b.total_cands]
        assert np.array_equal(got_mask, want_mask) and np.array_equal(got_rows, want_rows)
    assert store.device_status() == B.CCR_OK
    ws.free()
    store.free()


SWEEP = 256 * 256 * 4 * 16  # bytes of one round of the transfer kernel's grid
LIMIT = 16 << 20            # larger payloads go by copies


def _payload_bytes(n_req, n_cand, k):
    return n_req * k * 72 + 2 * 8 * (n_req + 1) + n_req * n_cand * 4 + n_req * 64


@pytest.mark.parametrize("entry", ["workspace", "static"])
@pytest.mark.parametrize("n_req,n_cand,k", [(2, 90_000, 300), (3, 500, 19_400), (3, 700, 24_800), (12, 16, 19_416), (12, 17, 19_416), (12, 18, 19_416)])
def test_payloads_around_the_sizes_of_the_transfer_kernel(n_req, n_cand, k, entry):
    """Pinned payloads of one and several rounds of the transfer kernel's grid, segments that lie across two rounds, up to and beyond its
    size limit, and a batch whose join is the warp-specialised one."""
    from paper_2609_22441_b200 import binding as B

    n_bytes = _payload_bytes(n_req, n_cand, k)
    assert {19_400: SWEEP < n_bytes < 1.1 * SWEEP, 24_800: SWEEP < n_bytes < 1.4 * SWEEP, 300: n_bytes < SWEEP}.get(k, True)
    assert k != 19_416 or {16: n_bytes < LIMIT, 17: n_bytes == LIMIT, 18: n_bytes > LIMIT}[n_cand]
    wls = [W.config1(seed=60 + i, n_docs=40_000 if k > 1000 else 200_000, n_req=n_req, n_cand=n_cand, edge_lo=k, edge_hi=k) for i in range(2)]
    wls[1].store = wls[0].store
    store = B.store_from_workload(wls[0])
    b, out_b = wls[0].batch, store.out_row_bytes(0)
    assert b.total_cands == n_req * n_cand and len(b.edge_keys) == n_req * k and b.edge_feats.nbytes == n_req * k * 64 and b.req_feats.nbytes == n_req * 64
    ws = B.Workspace(store, n_req, b.total_cands, len(b.edge_keys))
    names = ("edge_keys", "edge_feats", "edge_offsets", "cand_idx", "cand_offsets", "req_feats")
    bufs = [torch.zeros(getattr(b, n).nbytes, dtype=torch.uint8, pin_memory=True) for n in names]
    mask = torch.zeros(b.total_cands, dtype=torch.uint8, pin_memory=True)
    rows = torch.zeros((b.total_cands, out_b), dtype=torch.uint8)
    d_rows, d_mask = torch.zeros((b.total_cands, out_b), dtype=torch.uint8, device="cuda"), torch.zeros(b.total_cands, dtype=torch.uint8, device="cuda")
    for wl in wls:
        for n, buf in zip(names, bufs):
            buf.copy_(torch.from_numpy(np.ascontiguousarray(getattr(wl.batch, n)).reshape(-1).view(np.uint8)))
        args = (n_req, b.total_cands, k, n_req * k) + tuple(bufs)
        want_rows, want_mask = oracle.join_workload(wl, n_threads=4)
        if entry == "workspace":
            B.ccr_join_batch_host(store, ws, *args, rows, mask)
            torch.cuda.synchronize()
            got_rows, got_mask = rows.numpy(), mask.numpy()
        elif n_bytes > 16_770_000:  # with its roundings it does not fit the fixed block
            with pytest.raises(B.CcrError) as e:
                B.ccr_join_payload_static(store, *args, d_rows, d_mask)
            assert e.value.status == B.CCR_ERR_UNSUPPORTED
            continue
        else:
            B.ccr_join_payload_static(store, *args, d_rows, d_mask)
            torch.cuda.synchronize()
            got_rows, got_mask = d_rows.cpu().numpy(), d_mask.cpu().numpy()
        assert np.array_equal(got_mask, want_mask) and np.array_equal(got_rows, want_rows)
    assert store.device_status() == B.CCR_OK
    ws.free()
    store.free()


@pytest.mark.parametrize("n_req,n_cand", [(2, 900), (3, 262_200)])  # one group of requests, three pipelined ones
def test_a_workspace_of_another_store(n_req, n_cand):
    """A workspace serves any store whose rows fit its buffers; rows that do not are refused before anything is enqueued."""
    from paper_2609_22441_b200 import binding as B

    def workload(seed, edge_dim, req_dim):
        rng = np.random.default_rng(seed)
        st = W.make_store(rng, 40_000, 120_000, 8, np.float32)
        lists = [W.make_viewer(rng, 120_000, int(k), edge_dim, np.float16) for k in rng.integers(50, 700, size=n_req)]
        cands = [rng.integers(0, st.n_docs, size=n_cand).astype(np.int32) for _ in range(n_req)]
        req = rng.standard_normal((n_req, req_dim)).astype(np.float32)
        return W.Workload("w", seed, st, W.assemble_batch([k for k, _ in lists], [f for _, f in lists], cands, req, edge_dim, np.float16, req_dim, np.float32))

    def call(store, ws, wl, mask, rows):
        b = wl.batch
        B.ccr_join_batch_host(store, ws, b.n_req, b.total_cands, b.max_edge_len, int(b.edge_offsets[-1]), b.edge_keys, b.edge_feats.view(np.uint8), b.edge_offsets,
                              b.cand_idx, b.cand_offsets, b.req_feats, rows, mask)
        torch.cuda.synchronize()

    narrow, wide_req, wide_edge = workload(1, 8, 4), workload(2, 8, 24), workload(3, 64, 4)
    stores = {id(w): B.store_from_workload(w) for w in (narrow, wide_req, wide_edge)}
    mask = np.zeros(n_req * n_cand, np.uint8)
    big = B.Workspace(stores[id(wide_edge)], n_req, n_req * n_cand, max(int(w.batch.edge_offsets[-1]) for w in (narrow, wide_edge)))
    for wl in (narrow, wide_edge):
        rows = np.zeros((n_req * n_cand, stores[id(wl)].out_row_bytes(0)), np.uint8)
        call(stores[id(wl)], big, wl, mask, rows)
        want_rows, want_mask = oracle.join_workload(wl, n_threads=4)
        assert np.array_equal(mask, want_mask) and np.array_equal(rows, want_rows)
    # request rows of 96 bytes where 16 were sized for (the output rows fit), edge rows of 128 where 16 were
    small = B.Workspace(stores[id(narrow)], n_req, 64 * n_req * n_cand, 700 * n_req) if n_cand < 1000 else None
    for ws, wl in ((big, wide_req), (small, wide_edge)):
        if ws is None:
            continue
        rows = np.full((n_req * n_cand, stores[id(wl)].out_row_bytes(0)), 7, np.uint8)
        with pytest.raises(B.CcrError) as e:
            call(stores[id(wl)], ws, wl, mask, rows)
        assert e.value.status == B.CCR_ERR_INVALID_ARG and (rows == 7).all()
        ws.free()
    for st in stores.values():
        assert st.device_status() == B.CCR_OK
        st.free()
