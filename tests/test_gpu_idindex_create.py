"""ccr_idindex_create: indexes of different sizes and forms built by several threads at once."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_threads_build_indexes_of_different_sizes():
    """The build kernel's shared memory depends on the index; what one thread asks for must not be taken from another."""
    from paper_2609_22441_b200 import binding as B

    sizes = [3, 4_096, 100, 12_289, 900, 4_095]  # ids; regions from 3 ids to full ones
    failed = []

    def work(k):
        rng = np.random.default_rng(k)
        step = 1 << 31 if k % 2 else 5  # every other thread builds the form for ids that span more than 32 bits
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            for i in range(60):
                n = sizes[(i + k) % len(sizes)]
                ids = np.arange(n, dtype=np.int64) * step + 7
                q = torch.from_numpy(np.concatenate([ids[rng.integers(0, n, 50)], ids[:50] + 1])).cuda()
                stream.synchronize()
                try:
                    index = B.IdIndex(ids)
                    got = index.resolve(q).cpu().numpy()
                    index.free()
                    want = np.where((q.cpu().numpy() - 7) % step == 0, (q.cpu().numpy() - 7) // step, -1)
                    assert np.array_equal(got, want)
                except Exception as e:  # noqa: BLE001
                    failed.append("thread %d, %d ids: %r" % (k, n, e))
                    return

    threads = [threading.Thread(target=work, args=(k,)) for k in range(8)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed[:3]
