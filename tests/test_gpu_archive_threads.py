"""Archives of different table sizes rebuilt by several host threads at once,
each on its own stream: the kernels' shared-memory limit is one setting for
all of them, so every call must find it at what it needs."""
import ctypes
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def native():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2503_06763_gb300 import native
    return native


# interval, ids of each thread's archive: a warp per piece, a thread per piece
@pytest.mark.parametrize("K,ids", [(256, (3, 120, 160, 250)), (4096, (3, 40, 90, 250)), (64, (100, 200, 300, 390))])
def test_threads(native, K, ids):
    n, calls = 3000, 400
    lib = native.load()
    text = np.random.default_rng(1).integers(97, 101, n).astype(np.uint8)
    d_text = torch.from_numpy(text).cuda()
    jobs = []
    for j, n_ids in enumerate(ids):
        cols = np.random.default_rng(j).integers(0, n_ids, n + 1).astype(np.uint16)
        cols[7] = n_ids - 1
        arch = native.slpf_dfa_encode(cols, text, K)
        hdr = native.DfaHeader.from_buffer_copy(arch[:ctypes.sizeof(native.DfaHeader)].tobytes())
        assert hdr.n_ids == n_ids
        jobs.append((cols, hdr, torch.from_numpy(arch).cuda(), torch.zeros(n + 1, dtype=torch.int16, device="cuda"),
                     torch.full((1,), 7, dtype=torch.int32, device="cuda"), torch.cuda.Stream()))
    torch.cuda.synchronize()
    gate, codes = threading.Barrier(len(jobs)), [[] for _ in jobs]

    def work(j):
        _, hdr, arch, out, st, stream = jobs[j]
        torch.cuda.set_device(0)
        gate.wait()
        for _ in range(calls):
            codes[j].append(lib.re_slpf_dfa_decode(ctypes.byref(hdr), arch.data_ptr(), arch.numel(), d_text.data_ptr(),
                                                   out.data_ptr(), 2 * out.numel(), 2, st.data_ptr(),
                                                   ctypes.c_void_p(stream.cuda_stream)))

    threads = [threading.Thread(target=work, args=(j,)) for j in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert [c for per in codes for c in per if c] == []
    for cols, _, _, out, st, _ in jobs:
        assert int(st.item()) == 0
        assert np.array_equal(out.cpu().numpy().view(np.uint16), cols)
