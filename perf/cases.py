"""The work a serving program has this library do, as a list of cases that can be prepared, run and timed.

    single    one request per call, payload already on the device: the latency case
    batch     a ragged batch of requests in one call, first- or second-degree, any section widths
    host      the request payload arrives in host memory and is copied inside the call
    sort      affinity records that arrive unsorted are put in key order (Algorithm 1 step 1)
    resolve   document ids -> positions in the index (Eq. 6)
    flow      the whole device-side request: ids -> positions -> compaction -> sort -> padded join
    ingest    a batch of new documents is written into the store, then joined for the first time

Sizes are those of the benchmark configurations (`paper_2609_22441_b200/workloads.py`, `bench.py`) and of their
neighbourhood.  Inputs are drawn on the device with the same recipe: viewer keys are sorted samples of the author range,
a share `match` of a request's candidates are documents whose author (or engagers) are in the viewer's list, the rest
are drawn uniformly from the store.  List and request lengths depend on the case alone, so that every seed gives the
same shapes; which request gets which length depends on the seed.

Everything is moved and reduced bit for bit, so all outputs compare exactly.
"""
from __future__ import annotations

import numpy as np
import torch

from paper_2609_22441_b200 import binding as B
from paper_2609_22441_b200 import workloads as W

DEV = torch.device("cuda", 0)
CHUNK = 1 << 22          # document rows generated at a time
SINGLE_MAX_DOCS = 10_000_000
COS_FIRST, COS_DIM, COS_CHUNKS = 8, 50, 3   # the item embedding inside a document row, medoid chunks of a member


# ----------------------------------------------------------------------------------------------------------------
# cases
# ----------------------------------------------------------------------------------------------------------------
def _join(kind, **kw):
    case = dict(kind=kind, n_docs=1_000_000, authors_per_doc=5, n_req=64, n_cand=30_000, ragged=False, k_lo=50, k_hi=5000,
                k_dist="zipf", keys="uniform", match=0.5, unresolved=0.0, doc_dim=128, doc_dtype="float16", edge_dim=32,
                edge_dtype="float16", req_dim=16, engagers=False, first_only=False, cosine=False)
    case.update(kw)
    return case


def _production(kind, **kw):
    """The schema of the production-scale store: 128 fp16 features, engagers, 64 fp16 edge features, no request section."""
    base = dict(n_docs=50_000_000, authors_per_doc=1, n_req=256, n_cand=50_000, k_lo=10, k_hi=20_000, k_dist="log",
                match=0.7, edge_dim=64, req_dim=0, engagers=True)
    base.update(kw)
    return _join(kind, **base)


def listed():
    return [
        # the smallest request of the latency sweep: launch and dependent-read latency is all there is
        dict(_production("single", n_docs=SINGLE_MAX_DOCS, n_req=1, n_cand=1_000, k_lo=100, k_hi=100, first_only=True), name="single_1k"),
        # a large request of the sweep against a long edge list
        dict(_production("single", n_docs=SINGLE_MAX_DOCS, n_req=1, n_cand=50_000, k_lo=10_000, k_hi=10_000, first_only=True), name="single_50k"),
        # one request whose payload is in pinned host memory; rows stay on the device, the mask comes back
        dict(_join("host", n_req=1, k_lo=1000, k_hi=1000, k_dist="log", entry="workspace"), name="host_single"),
        # the headline batch: first-degree join, 64 requests x 30,000 candidates
        dict(_join("batch"), name="batch_first"),
        # the same shape with up to four engagers per document, looked up and reduced
        dict(_join("batch", engagers=True), name="batch_second"),
        # a deployment with other feature widths and dtypes, requests of very different lengths, ids handed out in
        # blocks, a few candidates the index does not know
        dict(_join("batch", n_docs=700_001, n_req=37, n_cand=17_003, ragged=True, keys="clustered", unresolved=0.02, doc_dim=104,
                   doc_dtype="float32", edge_dim=24, edge_dtype="float32", req_dim=20), name="batch_widths"),
        # production scale: 50M documents, 256 requests x 50,000 candidates in one launch
        dict(_production("batch", first_only=True), name="production_first"),
        dict(_production("batch"), name="production_second"),
        # unsorted affinity records of a production batch
        dict(kind="sort", n_req=256, k_lo=10, k_hi=20_000, k_dist="log", edge_dim=64, edge_dtype="float16", max_key=50_000_000, name="sort_production"),
        # ids of eight requests against a few hundred million indexed documents
        dict(kind="resolve", n_ids=300_000_000, n_queries=240_000, known=0.9, positions=False, name="resolve_8"),
        # the whole request flow with the derived cosine features
        dict(_join("flow", unresolved=0.03, cosine=True), name="flow"),
        # the bootstrap batch of ingestion and the first join over the new documents
        dict(_join("ingest", n_req=1, k_lo=1000, k_hi=1000, k_dist="log", n_cand=300_000, match=0.0, req_dim=0), name="ingest_300k"),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(lo * (hi / lo) ** rng.random()))))


def _draw_widths(rng):
    """Half of the deployments have the widths of the benchmark configurations, half have others."""
    if rng.random() < 0.5:
        return dict(doc_dim=128, doc_dtype="float16", edge_dim=rng.choice([32, 64]), edge_dtype="float16", req_dim=rng.choice([0, 16]))
    doc_dtype, edge_dtype = rng.choice(["float16", "float32"]), rng.choice(["float16", "float32"])
    return dict(doc_dim=8 * rng.randint(4, 24), doc_dtype=doc_dtype, edge_dim=8 * rng.randint(1, 8), edge_dtype=edge_dtype,
                req_dim=4 * rng.randint(0, 8))


def draw(rng):
    kind = rng.choice(["single", "single", "batch", "batch", "batch", "host", "sort", "resolve", "flow", "ingest"])
    if kind == "resolve":
        return dict(kind=kind, n_ids=_log_int(rng, 1_000_000, 300_000_000), n_queries=_log_int(rng, 1_000, 2_000_000),
                    known=round(rng.uniform(0.7, 1.0), 2), positions=rng.random() < 0.5)
    if kind == "sort":
        lo = _log_int(rng, 1, 200)
        return dict(kind=kind, n_req=_log_int(rng, 1, 256), k_lo=lo, k_hi=_log_int(rng, 2 * lo, 40_000), k_dist="log",
                    edge_dim=8 * rng.randint(1, 8), edge_dtype=rng.choice(["float16", "float32"]), max_key=_log_int(rng, 100_000, 1 << 40))
    c = _join(kind, n_docs=_log_int(rng, 100_000, SINGLE_MAX_DOCS), authors_per_doc=rng.choice([1, 2, 5]), match=round(rng.uniform(0.2, 0.8), 2),
              keys=rng.choice(["uniform", "uniform", "clustered"]), unresolved=rng.choice([0.0, 0.0, 0.03]), **_draw_widths(rng))
    # second-degree reduction is defined on float16 edge rows of at most 64 features
    c["engagers"] = c["edge_dtype"] == "float16" and rng.random() < 0.5
    c["first_only"] = c["engagers"] and rng.random() < 0.3
    c["k_dist"] = "log"
    c["k_lo"] = _log_int(rng, 1, 2_000)
    c["k_hi"] = _log_int(rng, c["k_lo"], 20_000)
    if kind == "single":
        c.update(n_req=1, n_cand=_log_int(rng, 100, 100_000))
        c["k_hi"] = c["k_lo"] = c["k_hi"]
    elif kind == "host":
        c.update(n_req=_log_int(rng, 1, 32), n_cand=_log_int(rng, 500, 30_000), ragged=True, entry=rng.choice(["workspace", "workspace", "static"]))
        if c["entry"] == "static":  # its payload goes through a fixed 16 MiB block
            c.update(n_req=min(c["n_req"], 4), k_lo=min(c["k_lo"], 5_000), k_hi=min(c["k_hi"], 5_000))
    elif kind == "ingest":
        c.update(n_req=1, n_cand=_log_int(rng, 1_000, 500_000), match=0.0, unresolved=0.0)
        c["k_hi"] = c["k_lo"] = c["k_hi"]
    else:
        c.update(n_req=_log_int(rng, 2, 256), n_cand=_log_int(rng, 300, 30_000), ragged=rng.random() < 0.7)
        if kind == "flow":
            c["cosine"] = c["doc_dtype"] == "float16" and c["doc_dim"] >= 64 and rng.random() < 0.7
    return c


# ----------------------------------------------------------------------------------------------------------------
# shapes (functions of the case alone)
# ----------------------------------------------------------------------------------------------------------------
def _edge_lengths(case):
    """Quantiles of the distribution, from a sample 64 times as long (so that a small batch is typical of it too)."""
    sampler = W.zipf_clipped_lengths if case["k_dist"] == "zipf" else W.log_uniform_lengths
    sample = sampler(case["k_lo"], case["k_hi"])(np.random.default_rng(case["n_req"]), 64 * case["n_req"])
    return np.sort(sample)[32::64]


def _cand_lengths(case):
    if not case["ragged"]:
        return np.full(case["n_req"], case["n_cand"], dtype=np.int64)
    rng = np.random.default_rng(case["n_req"] + 1)
    return np.maximum(1, np.rint(case["n_cand"] * rng.uniform(0.05, 1.95, case["n_req"]))).astype(np.int64)


def _flags(case):
    return (B.CCR_FLAG_FIRST_DEGREE_ONLY if case["first_only"] else 0) | (B.CCR_FLAG_COSINE if case["cosine"] else 0)


def _section_bytes(case):
    doc_b = case["doc_dim"] * np.dtype(case["doc_dtype"]).itemsize
    edge_b = case["edge_dim"] * np.dtype(case["edge_dtype"]).itemsize
    return doc_b, edge_b, case["req_dim"] * 4


# ----------------------------------------------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------------------------------------------
class _Draw:
    """Seeded draws on the device."""

    def __init__(self, seed):
        self.g = torch.Generator(device=DEV)
        self.g.manual_seed(int(seed))

    def ints(self, high, n, dtype=torch.int64):
        return torch.randint(0, int(high), (int(n),), generator=self.g, device=DEV, dtype=dtype)

    def unit(self, *shape):
        return torch.rand(shape, generator=self.g, device=DEV)

    def normal(self, rows, dim, dtype):
        return torch.randn((int(rows), int(dim)), generator=self.g, device=DEV).to(dtype)

    def permutation(self, n):
        return torch.randperm(int(n), generator=self.g, device=DEV)

    def shuffled(self, lengths):
        """The lengths in an order of this seed's own, on the device."""
        lengths = torch.from_numpy(np.ascontiguousarray(lengths)).to(DEV)
        return lengths[self.permutation(len(lengths))]


def _offsets(lengths):
    return torch.cat([torch.zeros(1, dtype=torch.int64, device=DEV), torch.cumsum(lengths, 0)])


def _owners(lengths):
    return torch.repeat_interleave(torch.arange(len(lengths), device=DEV), lengths)


def _viewer_keys(d, case, lengths, n_authors):
    """Per request an ascending list of distinct ids."""
    offsets, owner = _offsets(lengths), _owners(lengths)
    total = int(owner.numel())
    rank = torch.arange(total, device=DEV) - offsets[owner]
    if case["keys"] == "clustered":  # consecutive ids from a base of the viewer's own, one far outlier at the end
        base = d.ints(max(1, n_authors - int(lengths.max())), len(lengths))
        keys = base[owner] + rank
        last = offsets[1:][lengths > 1] - 1
        keys[last] = W.KEY_OUTLIER_BASE + d.ints(1 << 20, last.numel())
        return keys
    span = 1 << 34  # wider than any author range, so the requests' lists stay apart in one global sort
    keys = torch.sort(owner * span + d.ints(n_authors, total)).values
    step = torch.arange(total, device=DEV)
    keys = torch.cummax(keys - step, 0).values + step  # repeated draws become neighbouring ids
    return keys - owner * span


def _store_and_batch(d, case, extra_docs=0):
    """The store and one batch of requests: (store, tensors of the batch).  The store's last `extra_docs` rows stay
    unwritten (room for ingestion)."""
    n_docs, n_authors, n_req = case["n_docs"], case["n_docs"] * case["authors_per_doc"], case["n_req"]
    k_len, c_len = d.shuffled(_edge_lengths(case)), d.shuffled(_cand_lengths(case))
    edge_offsets, cand_offsets = _offsets(k_len), _offsets(c_len)
    keys = _viewer_keys(d, case, k_len, n_authors)
    edge_feats = d.unit(keys.numel(), case["edge_dim"]).to(getattr(torch, case["edge_dtype"]))
    req_feats = d.normal(n_req, case["req_dim"], torch.float32) if case["req_dim"] else None

    authors = d.ints(n_authors, n_docs)
    actors = types = None
    if case["engagers"]:
        slot = torch.arange(W.MAX_ACTOR_SLOTS, device=DEV)
        count = torch.poisson(torch.full((n_docs, 1), 1.5, device=DEV), generator=d.g)
        actors = torch.where(slot < count, d.ints(n_authors, n_docs * W.MAX_ACTOR_SLOTS).view(n_docs, -1), -1)
        types = torch.randint(0, W.ENGAGEMENT_TYPES, actors.shape, generator=d.g, device=DEV, dtype=torch.uint8)
        del count

    # documents of a viewer's network: their author (with engagers: the author or some of the engagers) is in the list
    forced_len = torch.minimum((case["match"] * c_len).to(torch.int64), torch.tensor(n_docs // n_req, device=DEV))
    owner = _owners(forced_len)
    docs = d.permutation(n_docs)[:owner.numel()]

    def pick(n_slots):
        u = d.unit(owner.numel(), n_slots)
        return keys[edge_offsets[owner][:, None] + torch.minimum((u * k_len[owner][:, None]).to(torch.int64), k_len[owner][:, None] - 1)]

    if not case["engagers"]:
        authors[docs] = pick(1)[:, 0]
    else:
        mine = actors[docs]
        by_author = (mine[:, 0] < 0) | (d.unit(docs.numel()) < 0.5)
        authors[docs] = torch.where(by_author, pick(1)[:, 0], authors[docs])
        hit = (d.unit(*mine.shape) < 0.6) & (mine >= 0)
        actors[docs] = torch.where(hit, pick(W.MAX_ACTOR_SLOTS), mine)

    natural_len = c_len - forced_len
    cand = torch.cat([docs, d.ints(n_docs, int(natural_len.sum()))])
    request = torch.cat([owner, _owners(natural_len)])
    order = torch.argsort(request * (1 << 32) + d.ints(1 << 32, request.numel()))
    cand = cand[order].to(torch.int32)
    if case["unresolved"] > 0:
        cand = torch.where(d.unit(cand.numel()) < case["unresolved"], -1, cand)
    del order, request, docs, owner

    store = B.Docstore(n_docs + extra_docs, case["doc_dim"], case["doc_dtype"], case["edge_dim"], case["edge_dtype"], case["req_dim"], "float32",
                       W.MAX_ACTOR_SLOTS if case["engagers"] else 0, _sum_mask(case))
    store.upload(0, None, authors, actors, types)
    for first in range(0, n_docs, CHUNK):
        store.upload(first, d.normal(min(CHUNK, n_docs - first), case["doc_dim"], getattr(torch, case["doc_dtype"])))
    torch.cuda.synchronize(DEV)  # the sources of the uploads may go now
    batch = dict(n_req=n_req, total=int(cand.numel()), max_edge_len=int(k_len.max()), n_max=int(c_len.max()), edge_keys=keys, edge_feats=edge_feats,
                 edge_offsets=edge_offsets, cand_idx=cand, cand_offsets=cand_offsets, req_feats=req_feats)
    return store, batch


def _sum_mask(case):
    """The upper half of every 32 edge features are counts (summed over the engagers), the lower half recencies (maximum)."""
    return (W.SUM_DIMS_16_31 | (W.SUM_DIMS_16_31 << 32)) if case["engagers"] else 0


def _outputs(store, case, rows):
    return (torch.empty((rows, store.out_row_bytes(_flags(case))), dtype=torch.uint8, device=DEV),
            torch.empty((rows,), dtype=torch.uint8, device=DEV))


def _shuffle_lists(d, b):
    """The records of every list in random order, as a payload brings them."""
    owner = _owners(b["edge_offsets"][1:] - b["edge_offsets"][:-1])
    order = torch.argsort(owner * (1 << 32) + d.ints(1 << 32, owner.numel()))
    return b["edge_keys"][order].contiguous(), b["edge_feats"][order].contiguous()


class _WorkspaceRows:
    """The output rows of a workspace as something torch can wrap; the tensor keeps this object, and with it the
    workspace, alive."""

    def __init__(self, ws, n_bytes):
        self.ws = ws
        self.__cuda_array_interface__ = {"shape": (n_bytes,), "typestr": "|u1", "data": (ws.outputs()[0], False), "version": 3}


def prepare(case, seed):
    return _PREPARE[case["kind"]](case, _Draw(seed))


def _prepare_join(case, d):
    store, b = _store_and_batch(d, case)
    rows, mask = _outputs(store, case, b["total"])
    return dict(b, case=case, store=store, rows=rows, mask=mask, flags=_flags(case))


def _prepare_host(case, d):
    store, b = _store_and_batch(d, case)
    pinned = {k: v.cpu().pin_memory() for k, v in b.items() if isinstance(v, torch.Tensor)}
    state = dict(b, **pinned)
    state.update(case=case, store=store, flags=_flags(case), total_edges=int(pinned["edge_keys"].numel()))
    if case["entry"] == "static":
        state["rows"], state["mask"] = _outputs(store, case, b["total"])
    else:
        ws = B.Workspace(store, b["n_req"], b["total"], state["total_edges"])
        n_bytes = b["total"] * store.out_row_bytes(_flags(case))
        state.update(ws=ws, rows=torch.as_tensor(_WorkspaceRows(ws, n_bytes), device=DEV), mask=torch.empty(b["total"], dtype=torch.uint8).pin_memory())
    return state


def _prepare_sort(case, d):
    lengths = d.shuffled(_edge_lengths(case))
    n = int(lengths.sum())
    feats = d.unit(n, case["edge_dim"]).to(getattr(torch, case["edge_dtype"]))
    keys = d.ints(case["max_key"], n)
    store = B.Docstore(16, 8, "float16", case["edge_dim"], case["edge_dtype"])
    return dict(case=case, store=store, n_req=case["n_req"], max_edge_len=int(lengths.max()), keys_in=keys, feats_in=feats, edge_offsets=_offsets(lengths),
                keys=torch.empty_like(keys), feats=torch.empty_like(feats), perm=torch.empty(n, dtype=torch.int32, device=DEV))


def _prepare_resolve(case, d):
    ids = 2 * torch.cumsum(1 + d.ints(3, case["n_ids"]), 0)
    positions = d.permutation(case["n_ids"]).to(torch.int32) if case["positions"] else None
    index = B.IdIndex(ids, positions)
    queries = ids[d.ints(case["n_ids"], case["n_queries"])]
    queries = torch.where(d.unit(case["n_queries"]) < case["known"], queries, queries + 1)
    return dict(case=case, index=index, queries=queries, pos=torch.empty(case["n_queries"], dtype=torch.int32, device=DEV))


def _prepare_flow(case, d):
    store, b = _store_and_batch(d, case)
    if case["cosine"]:
        store.set_cosine(COS_FIRST, COS_DIM, COS_CHUNKS)
    ids = 10 * torch.arange(case["n_docs"], device=DEV) + d.ints(10, case["n_docs"])
    owner = d.permutation(case["n_docs"]).to(torch.int32)  # document that holds the id of each rank
    index = B.IdIndex(ids, owner)
    id_of = torch.empty_like(ids)
    id_of[owner.to(torch.int64)] = ids
    known = b["cand_idx"] >= 0
    queries = torch.where(known, id_of[b["cand_idx"].clamp(min=0).to(torch.int64)], -5)
    keys_in, feats_in = _shuffle_lists(d, b)
    member = d.normal(b["n_req"], COS_CHUNKS * COS_DIM, torch.float16) if case["cosine"] else None
    C = b["total"]
    out_b = store.out_row_bytes(_flags(case))
    state = dict(b, case=case, store=store, index=index, queries=queries, keys_in=keys_in, feats_in=feats_in, member=member, flags=_flags(case),
                 pos=torch.empty(C, dtype=torch.int32, device=DEV), perm=torch.empty(keys_in.numel(), dtype=torch.int32, device=DEV),
                 keys=torch.empty_like(keys_in), feats=torch.empty_like(feats_in), offs=torch.empty(b["n_req"] + 1, dtype=torch.int64, device=DEV),
                 rows=torch.empty((b["n_req"], b["n_max"], out_b), dtype=torch.uint8, device=DEV),
                 mask=torch.empty((b["n_req"], b["n_max"]), dtype=torch.uint8, device=DEV))
    # entries behind the last valid candidate are never written by the compaction
    state["kept"], state["src"] = (torch.full((C,), -1, dtype=torch.int32, device=DEV) for _ in range(2))
    return state


def _prepare_ingest(case, d):
    n = case["n_cand"]
    store, b = _store_and_batch(d, case, extra_docs=2 * n)
    # the new documents' positions, as the host assigned them: scattered over the free rows; half are by authors the viewer knows
    positions = (case["n_docs"] + d.permutation(2 * n)[:n]).to(torch.int32)
    known = b["edge_keys"][d.ints(b["edge_keys"].numel(), n)]
    authors = torch.where(d.unit(n) < 0.5, known, d.ints(case["n_docs"] * case["authors_per_doc"], n))
    actors = types = None
    if case["engagers"]:
        actors = torch.where(d.unit(n, W.MAX_ACTOR_SLOTS) < 0.3, known[:, None], -1)
        types = torch.randint(0, W.ENGAGEMENT_TYPES, actors.shape, generator=d.g, device=DEV, dtype=torch.uint8)
    rows, mask = _outputs(store, case, n)
    b["cand_idx"] = positions[d.permutation(n)].contiguous()
    return dict(b, case=case, store=store, positions=positions, new_rows=d.normal(n, case["doc_dim"], getattr(torch, case["doc_dtype"])), authors=authors,
                actors=actors, types=types, rows=rows, mask=mask, flags=_flags(case))


_PREPARE = {"single": _prepare_join, "batch": _prepare_join, "host": _prepare_host, "sort": _prepare_sort, "resolve": _prepare_resolve,
            "flow": _prepare_flow, "ingest": _prepare_ingest}


# ----------------------------------------------------------------------------------------------------------------
# one pass
# ----------------------------------------------------------------------------------------------------------------
def _words(rows):
    """Output rows (whole 16-byte pieces) as 64-bit words."""
    return rows.view(torch.int64)


def run(state):
    return _RUN[state["case"]["kind"]](state)


def _run_join(s):
    B.ccr_join_batch(s["store"], s["n_req"], s["total"], s["max_edge_len"], s["edge_keys"], s["edge_feats"], s["edge_offsets"], s["cand_idx"],
                     s["cand_offsets"], s["req_feats"], s["rows"], s["mask"], s["flags"])
    return {"rows": _words(s["rows"]), "mask": s["mask"]}


def _run_host(s):
    payload = (s["n_req"], s["total"], s["max_edge_len"], s["total_edges"], s["edge_keys"], s["edge_feats"], s["edge_offsets"], s["cand_idx"],
               s["cand_offsets"], s["req_feats"])
    if s["case"]["entry"] == "static":
        B.ccr_join_payload_static(s["store"], *payload, s["rows"], s["mask"], s["flags"])
    else:
        B.ccr_join_batch_host(s["store"], s["ws"], *payload, None, s["mask"], s["flags"])
    return {"rows": _words(s["rows"]), "mask": s["mask"]}


def _run_sort(s):
    B.ccr_sort_edges(s["store"], s["n_req"], s["max_edge_len"], s["keys_in"], s["feats_in"], s["edge_offsets"], s["keys"], s["feats"], s["perm"])
    return {"keys": s["keys"], "feats": s["feats"].view(torch.int32), "perm": s["perm"]}


def _run_resolve(s):
    return {"pos": s["index"].resolve(s["queries"], s["pos"])}


def _run_flow(s):
    s["index"].resolve(s["queries"], s["pos"])
    B.ccr_compact_valid(s["store"], s["n_req"], s["total"], s["pos"], s["cand_offsets"], s["kept"], s["offs"], s["src"])
    B.ccr_sort_edges(s["store"], s["n_req"], s["max_edge_len"], s["keys_in"], s["feats_in"], s["edge_offsets"], s["keys"], s["feats"], s["perm"])
    B.ccr_join_batch_ex(s["store"], s["n_req"], s["total"], s["max_edge_len"], s["keys"], s["feats"], s["edge_offsets"], s["kept"], s["offs"],
                        s["req_feats"], s["rows"], s["mask"], s["flags"], None, s["n_max"], s["member"])
    return {"rows": _words(s["rows"]), "mask": s["mask"], "offsets": s["offs"], "kept": s["kept"], "src": s["src"]}


def _run_ingest(s):
    s["store"].upsert(s["positions"], s["new_rows"], s["authors"], s["actors"], s["types"])
    return _run_join(s)


_RUN = {"single": _run_join, "batch": _run_join, "host": _run_host, "sort": _run_sort, "resolve": _run_resolve, "flow": _run_flow, "ingest": _run_ingest}


# ----------------------------------------------------------------------------------------------------------------
# what a pass cannot do without
# ----------------------------------------------------------------------------------------------------------------
def _distinct(n_values, n_draws):
    """Expected number of distinct values among uniform draws."""
    return n_values * -np.expm1(n_draws * np.log1p(-1.0 / n_values)) if n_values > 1 else min(n_values, n_draws)


def _join_bytes(case):
    """Every distinct document row, id (record) and matched edge row read once, the keys, positions and offsets read
    once, every output row and mask byte written once.  The pairing of list and request lengths is the seed's: the
    mean list stands for all."""
    doc_b, edge_b, req_b = _section_bytes(case)
    k_len, c_len = _edge_lengths(case), _cand_lengths(case)
    C, n_req = float(c_len.sum()), case["n_req"]
    second = case["engagers"] and not case["first_only"]
    valid = C * (1.0 - case["unresolved"])
    forced = min(case["match"] * C, case["n_docs"])
    docs = forced + _distinct(case["n_docs"], C - forced) * (1.0 - forced / case["n_docs"])
    if case["kind"] == "ingest":
        docs = C
    matches = (1.8 if second else (0.65 if case["engagers"] else 1.0)) * (0.5 * C if case["kind"] == "ingest" else forced)
    matched = n_req * float(np.mean([_distinct(k, matches / n_req) for k in k_len]))
    out_b = doc_b + edge_b * (2 if second else 1) + req_b + (32 if case["cosine"] else 0)
    out_rows = n_req * float(c_len.max()) if case["kind"] == "flow" else C
    return (docs * (valid / C) * (doc_b + (64 if second else 8)) + matched * edge_b + 8.0 * k_len.sum() + 4.0 * C + n_req * (req_b + 32.0) + out_rows * (out_b + 1))


def _sort_bytes(case):
    n = float(_edge_lengths(case).sum())
    return n * (2 * (8 + case["edge_dim"] * np.dtype(case["edge_dtype"]).itemsize) + 4)


def work(case):
    kind = case["kind"]
    if kind == "sort":
        total = _sort_bytes(case)
    elif kind == "resolve":
        total = case["n_queries"] * (8.0 + 8.0 + 4.0 + (4.0 if case["positions"] else 0.0))
    else:
        total = _join_bytes(case)
        if kind == "flow":  # ids in, positions, kept positions and source indices out, the sort
            total += float(_cand_lengths(case).sum()) * (8 + 8 + 4 + 4 + 8) + _sort_bytes(case)
        if kind == "ingest":  # the batch is read and its rows are written
            total += case["n_cand"] * (2.0 * (_section_bytes(case)[0] + (64 if case["engagers"] else 8)) + 4)
    return {"bytes": float(total), "flops": 0.0}


def tolerance(case):
    return "exact"
