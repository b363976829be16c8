"""GPU parity of ccr_resolve_ids where there are levels below the top one: the sizes at which a level is added (2,048 keys of the top level,
a factor of 8 for each level below it, 4,096 ids per region), in both forms of the buckets, from the device and from the host."""
import numpy as np
import pytest

from oracle import oracle

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

TWO_LEVELS = 2_049 * 4_096 + 1         # one region more than the top level can tell apart
THREE_LEVELS = 16_392 * 4_096 + 1
REGION = 4_096


@pytest.mark.parametrize("wide", [False, True])
@pytest.mark.parametrize("n_ids,on_device", [(TWO_LEVELS - 1, True), (TWO_LEVELS, True), (TWO_LEVELS, False), (TWO_LEVELS + 8 * REGION + 77, True),
                                             (THREE_LEVELS - 1, True), (THREE_LEVELS, True)])
def test_sizes_at_which_a_level_is_added(n_ids, on_device, wide):
    from paper_2609_22441_b200 import binding as B

    gen = torch.Generator(device="cuda")
    gen.manual_seed(n_ids + wide)
    # steps of about 2^36 where a region must not fit 32 bits, negative ids first
    ids = torch.randint(1, 1 << 37 if wide else 4, (n_ids,), generator=gen, device="cuda")
    ids = torch.cumsum(ids, 0) - (1 << (60 if wide else 10))
    host = ids.cpu().numpy()
    rng = np.random.default_rng(n_ids)
    n_regions = -(-n_ids // REGION)
    per_region = -(-n_ids // n_regions)
    pos = rng.permutation(n_ids).astype(np.int32) if n_ids < THREE_LEVELS - 1 else None
    ends = np.arange(per_region - 1, n_ids, per_region)
    edges = np.concatenate([ends, np.minimum(ends + 1, n_ids - 1), [0, n_ids - 1, n_ids // 2]])
    some = host[np.concatenate([edges, rng.integers(0, n_ids, size=200_000)])]
    q = np.concatenate([some, some + 1, some[:50_000] - 1, some[:50_000] + (1 << 32), [np.iinfo(np.int64).min, np.iinfo(np.int64).max, host[0] - 1, host[-1] + 1]])
    index = B.IdIndex(ids if on_device else host, None if pos is None else (torch.from_numpy(pos).cuda() if on_device else pos))
    got = index.resolve(torch.from_numpy(q).cuda()).cpu().numpy()
    assert np.array_equal(got, oracle.resolve_ids(host, q, pos))
    index.free()
