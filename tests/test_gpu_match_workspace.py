"""Match extraction in a workspace without room for the spans of the counting
pass: the same pairs; one byte group less is refused."""
import ctypes

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def native():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2503_06763_gb300 import native
    return native


def _up(v):
    return -(-v // 256) * 256


@pytest.mark.parametrize("n", [0, 1, 2047, 2048, 70_001, (1 << 21) + 9])
def test_counts_alone(native, n):
    rx = native.Regex(W.AB_RE)
    t = torch.from_numpy(W.ab_text(max(n, 1), seed=4)[:n].copy()).cuda()
    cols, st, kind = rx.parse(t)
    want, total = rx.matches(cols, st, n, 5, kind)                  # every "ab"
    tiles = n // 2048 + 1
    size = _up(8 * tiles) + _up(8 * -(-tiles // 1024))
    lib, cb = native.load(), cols.element_size()
    slpf = native.Slpf(native.KINDS[kind], cb, n + 1, cols.data_ptr(), cols.numel() * cb, st.data_ptr())
    for room, cap in ((size, total), (size, total // 2), (size + 256, total), (size - 256, total)):
        ws = torch.empty(max(room, 1), dtype=torch.uint8, device="cuda")
        pairs = torch.full((max(cap, 1), 2), -1, dtype=torch.int64, device="cuda")
        count = torch.full((1,), -1, dtype=torch.int64, device="cuda")
        rc = lib.re_matches(rx._h, ctypes.byref(slpf), n, 5, pairs.data_ptr(), cap, count.data_ptr(), ws.data_ptr(), room,
                            ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        torch.cuda.synchronize()
        if room < size:
            assert rc == -8
            continue
        assert rc == 0 and int(count.item()) == total
        assert np.array_equal(pairs[:cap].cpu().numpy(), want[:cap].cpu().numpy())
