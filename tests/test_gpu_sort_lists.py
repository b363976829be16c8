"""GPU parity of the whole-list radix sort (ccr_sort_edges, lists of up to 32,768 records) against the CPU oracle: list
lengths around a block's and a cluster's share, key ranges around every rule of the kernel (no differing bit, one digit,
just room and no room for the index, full 64 bits), with and without the permutation output."""
import numpy as np
import pytest

from oracle import oracle
from paper_2609_22441_b200 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

IMIN, IMAX = np.iinfo(np.int64).min, np.iinfo(np.int64).max
LENS = ([1, 0, 2, 127, 128, 129, 511, 512], [513, 1023, 1024, 1025, 300], [4095, 4096, 4097, 1, 8191], [8193, 12_288, 12_289, 1000, 255], [32_768, 32_767, 20_000, 5, 28_673])
KEYS = {
    "equal": lambda rng, n: np.full(n, 7_000_000_019, np.int64),
    "few": lambda rng, n: rng.integers(0, 3, size=n),
    "26_bits": lambda rng, n: rng.integers(0, 50_000_000, size=n),
    "48_bits": lambda rng, n: rng.integers(0, 1 << 48, size=n),  # with 15 index bits: just room
    "49_bits": lambda rng, n: rng.integers(0, 1 << 49, size=n),
    "high_half": lambda rng, n: rng.integers(0, 5, size=n) << 61,  # only the upper word differs
    "outlier": lambda rng, n: np.where(np.arange(n) == n // 2, IMAX - 3, 123_456_789 + rng.permutation(n)),
    "any": lambda rng, n: rng.integers(IMIN, IMAX, size=n, endpoint=True),
    "ends": lambda rng, n: np.array([IMIN, -1, 0, IMAX])[rng.integers(0, 4, size=n)],
}


@pytest.mark.parametrize("with_perm", [True, False])
@pytest.mark.parametrize("kind", list(KEYS))
@pytest.mark.parametrize("lens", LENS, ids=lambda l: str(max(l)))
def test_whole_lists_match_the_oracle(lens, kind, with_perm):
    from paper_2609_22441_b200 import binding as B

    if not with_perm and max(lens) > 19_000:
        pytest.skip("refused without a permutation output")
    rng = np.random.default_rng(len(kind) + sum(lens))
    keys = np.concatenate([KEYS[kind](rng, n) for n in lens]).astype(np.int64)
    feats = rng.integers(0, 1 << 16, size=(len(keys), 24), dtype=np.uint16).view(np.float16)  # 48-byte rows
    eo = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    want_k, want_f, want_p = oracle.sort_edges(keys, feats, eo)
    store = B.Docstore(16, 8, "float16", 24, "float16")
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()
    k_out = torch.full((len(keys) + 2,), -7, dtype=torch.int64, device="cuda")
    f_out = torch.full((len(keys) + 2, 24), 7.0, dtype=torch.float16, device="cuda")
    p_out = torch.full((len(keys) + 2,), -7, dtype=torch.int32, device="cuda")
    n = len(keys)
    B.ccr_sort_edges(store, len(lens), max(lens), dev(keys), dev(feats.view(np.int16)), dev(eo), k_out[1:-1], f_out, p_out[1:-1] if with_perm else None)
    torch.cuda.synchronize()
    assert np.array_equal(k_out.cpu().numpy()[1:-1], want_k) and int(k_out[0]) == -7 and int(k_out[-1]) == -7
    assert np.array_equal(f_out.cpu().numpy()[:n].view(np.uint16), want_f.view(np.uint16)) and bool((f_out[n:] == 7).all())
    if with_perm:
        assert np.array_equal(p_out.cpu().numpy()[1:-1], want_p) and int(p_out[0]) == -7 and int(p_out[-1]) == -7
    store.free()


def test_a_longer_batch_with_keys_that_cannot_be_packed():
    """A list beyond the clusters' reach sends the batch to the chunked path; negative and far keys take its fallback."""
    from paper_2609_22441_b200 import binding as B

    rng = np.random.default_rng(3)
    lens = [40_000, 9_000, 100, 0, 33_000]
    keys = np.concatenate([KEYS[k](rng, n) for k, n in zip(("any", "26_bits", "few", "equal", "ends"), lens)]).astype(np.int64)
    feats = rng.integers(0, 1 << 16, size=(len(keys), 24), dtype=np.uint16).view(np.float16)
    eo = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    want_k, want_f, want_p = oracle.sort_edges(keys, feats, eo)
    store = B.Docstore(16, 8, "float16", 24, "float16")
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()
    k_out, p_out = torch.empty(len(keys), dtype=torch.int64, device="cuda"), torch.empty(len(keys), dtype=torch.int32, device="cuda")
    f_out = torch.empty((len(keys), 24), dtype=torch.float16, device="cuda")
    B.ccr_sort_edges(store, len(lens), max(lens), dev(keys), dev(feats.view(np.int16)), dev(eo), k_out, f_out, p_out)
    torch.cuda.synchronize()
    assert np.array_equal(k_out.cpu().numpy(), want_k) and np.array_equal(p_out.cpu().numpy(), want_p)
    assert np.array_equal(f_out.cpu().numpy().view(np.uint16), want_f.view(np.uint16))
    store.free()


def test_many_long_lists_of_equal_keys():
    """Lists of several blocks without a differing bit are sorted without a single pass: the blocks of a cluster only exchange what
    differs and then leave at different times (a last block of one record beside full ones).  One list of each length has a
    differing bit in its last record."""
    from paper_2609_22441_b200 import binding as B

    rng = np.random.default_rng(11)
    lens = [n for n in (4097, 8191, 8193, 12_289, 16_385, 28_673, 32_768) for _ in range(24)]
    keys = [np.full(n, 3 * i - 200, np.int64) for i, n in enumerate(lens)]
    for i in range(0, len(lens), 24):
        keys[i][-1] -= 1
    keys = np.concatenate(keys)
    feats = rng.integers(0, 1 << 16, size=(len(keys), 8), dtype=np.uint16).view(np.float16)
    eo = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    want_k, want_f, want_p = oracle.sort_edges(keys, feats, eo)
    store = B.Docstore(16, 8, "float16", 8, "float16")
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()
    k_in, f_in, o = dev(keys), dev(feats.view(np.int16)), dev(eo)
    for _ in range(5):
        k_out, p_out = torch.full_like(k_in, -7), torch.full((len(keys),), -7, dtype=torch.int32, device="cuda")
        f_out = torch.empty((len(keys), 8), dtype=torch.float16, device="cuda")
        B.ccr_sort_edges(store, len(lens), max(lens), k_in, f_in, o, k_out, f_out, p_out)
        torch.cuda.synchronize()
        assert np.array_equal(k_out.cpu().numpy(), want_k) and np.array_equal(p_out.cpu().numpy(), want_p)
        assert np.array_equal(f_out.cpu().numpy().view(np.uint16), want_f.view(np.uint16))
    store.free()


@pytest.mark.parametrize("rows_of", [5, 10_000])  # few distinct keys (equal ones keep their order), hardly an equal pair
@pytest.mark.parametrize("kind", ["both_halves", "same_low", "same_high"])
def test_short_lists_of_wide_keys(kind, rows_of):
    """Keys that leave no room for the index in lists up to the length of the register network: sorted by halves."""
    from paper_2609_22441_b200 import binding as B

    rng = np.random.default_rng(rows_of)
    lens = [2, 31, 33, 127, 128, 129, 300, 512, 513, 1023, 1024, 1, 0, 1025]
    pool = rng.integers(IMIN, IMAX, size=rows_of, endpoint=True)
    if kind == "same_low":
        pool = pool & ~np.int64(0xffffffff) | 77
    if kind == "same_high":
        pool = pool & np.int64(0xffffffff) | np.int64(5 << 40)
        pool[::2] |= np.int64(1 << 62)
    keys = np.concatenate([pool[rng.integers(0, rows_of, size=n)] for n in lens]).astype(np.int64)
    feats = rng.integers(0, 1 << 16, size=(len(keys), 8), dtype=np.uint16).view(np.float16)
    eo = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    want_k, want_f, want_p = oracle.sort_edges(keys, feats, eo)
    store = B.Docstore(16, 8, "float16", 8, "float16")
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()
    k_in = dev(keys)
    for bound in (1024, max(lens)):  # the last list is cut at the smaller bound
        k_out, p_out, f_out = torch.full_like(k_in, -7), torch.full((len(keys),), -7, dtype=torch.int32, device="cuda"), torch.zeros((len(keys), 8), dtype=torch.float16, device="cuda")
        B.ccr_sort_edges(store, len(lens), bound, k_in, dev(feats.view(np.int16)), dev(eo), k_out, f_out, p_out)
        torch.cuda.synchronize()
        n = len(keys) if bound > 1024 else len(keys) - 1025
        assert np.array_equal(k_out.cpu().numpy()[:n], want_k[:n]) and np.array_equal(p_out.cpu().numpy()[:n], want_p[:n])
        assert np.array_equal(f_out.cpu().numpy()[:n].view(np.uint16), want_f[:n].view(np.uint16))
        assert bound > 1024 or int(k_out[-1]) == -7
    store.free()


@pytest.mark.parametrize("bits", [33, 47, 64])
@pytest.mark.parametrize("lens", [[1025, 1030, 4096, 4095], [4097, 8192, 5000], [12_289, 32_768, 20_001]], ids=lambda l: str(max(l)))
def test_keys_that_share_a_prefix(lens, bits):
    """Spread keys are sorted by a prefix of three digits and the records that share one are put in order behind it.  Per list a run
    of such records at a place of its own, across the border of two blocks among others: none, of two, the longest that is put in order (65)
    and the shortest that is not, with equal keys among them; wide keys that differ only below the bits that fit a word."""
    from paper_2609_22441_b200 import binding as B

    rng = np.random.default_rng(bits + max(lens))

    def keys_of(n, run, at, fine):
        top = 1 << (min(bits, 63) - 1)
        keys = rng.integers(0, 2 * top - 1, size=n, dtype=np.int64)
        keys[0], keys[1] = 0, 2 * top - 1  # the range is used up to its ends
        s = np.sort(keys)
        base = int(s[min(at, n - 1)]) >> 14 << 14
        where = rng.choice(n - 2, size=run, replace=False) + 2
        keys[where] = base + rng.integers(0, 1 << (6 if fine else 14), size=run)
        if bits == 64:
            keys = np.where(rng.random(n) < 0.5, keys, -keys)
        return keys

    cases = [(n, run, at, fine) for n in lens for run in (0, 2, 40, 65, 66, 150) for at, fine in ((n // 2, False), (4096 - 20, True), (n - 5, False))]
    keys = np.concatenate([keys_of(*c) for c in cases])
    lens_all = [c[0] for c in cases]
    feats = rng.integers(0, 1 << 16, size=(len(keys), 8), dtype=np.uint16).view(np.float16)
    eo = np.concatenate([[0], np.cumsum(lens_all)]).astype(np.int64)
    want_k, want_f, want_p = oracle.sort_edges(keys, feats, eo)
    store = B.Docstore(16, 8, "float16", 8, "float16")
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()
    k_in, f_in, o = dev(keys), dev(feats.view(np.int16)), dev(eo)
    for with_perm in (True, False):
        if not with_perm and max(lens) > 19_000:
            continue
        k_out, p_out, f_out = torch.full_like(k_in, -7), torch.full((len(keys),), -7, dtype=torch.int32, device="cuda"), torch.zeros((len(keys), 8), dtype=torch.float16, device="cuda")
        B.ccr_sort_edges(store, len(lens_all), max(lens), k_in, f_in, o, k_out, f_out, p_out if with_perm else None)
        torch.cuda.synchronize()
        assert np.array_equal(k_out.cpu().numpy(), want_k) and (not with_perm or np.array_equal(p_out.cpu().numpy(), want_p))
        assert np.array_equal(f_out.cpu().numpy().view(np.uint16), want_f.view(np.uint16))
    store.free()
