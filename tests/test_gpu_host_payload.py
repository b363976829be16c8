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
