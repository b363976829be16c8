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


@pytest.mark.parametrize("on_device", [False, True])
def test_a_call_that_fails_says_why(on_device):
    """A refused runtime call (no allocation is allowed while a stream of this thread is being captured) is a CUDA error, not a lack of memory;
    a table that does not fit what is free is."""
    import ctypes

    from paper_2609_22441_b200 import binding as B

    ids = torch.arange(20_000_000, dtype=torch.int64) * 3
    ids = ids.cuda() if on_device else ids
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    driver, graph = ctypes.CDLL("libcuda.so.1"), ctypes.c_void_p()
    assert driver.cuStreamBeginCapture_v2(ctypes.c_void_p(stream.cuda_stream), 0) == 0
    try:
        with pytest.raises(B.CcrError) as e:
            B.IdIndex(ids[:1_000])
    finally:
        driver.cuStreamEndCapture(ctypes.c_void_p(stream.cuda_stream), ctypes.byref(graph))
    assert e.value.status == B.CCR_ERR_CUDA
    torch.cuda.empty_cache()
    filler = torch.empty(torch.cuda.mem_get_info()[0] - (128 << 20), dtype=torch.uint8, device="cuda")  # 128 MB are left, the table needs 320
    try:
        with pytest.raises(B.CcrError) as e:
            B.IdIndex(ids)
    finally:
        del filler
        torch.cuda.empty_cache()
    assert e.value.status == B.CCR_ERR_OOM
    index = B.IdIndex(ids)
    q = torch.tensor([0, 1, 3, 59_999_997], device="cuda")
    assert index.resolve(q).cpu().tolist() == [0, -1, 1, 19_999_999]
    index.free()
