"""Match extraction where its tiles can go wrong: texts that end on and around
a 512-column subtile and a 2048-column tile, tiles with more spans than their
records hold, spans too long for a record, columns at an address that is not a
multiple of 16, and a capacity inside a tile; against closed forms."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def lib():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2503_06763_gb300 import Regex
    return Regex


@pytest.mark.parametrize("n", [511, 512, 513, 2047, 2048, 2049, 2048 * 3 + 511, 70_001])
@pytest.mark.parametrize("kind", ["dense", "dict"])
@pytest.mark.parametrize("period", [2, 7, 9, 40])
def test_ab_spans(lib, n, kind, period):
    """Group 5 of (a|b|ab)* is every "ab": period 2 and 7 put more than 256 of
    them in a tile of 2048 columns, 9 and 40 fewer."""
    rx = lib(W.AB_RE)
    host = np.full(n, ord("b"), dtype=np.uint8)
    host[::period] = ord("a")
    t = torch.from_numpy(host).cuda()
    cols, st, k = rx.parse(t, kind=kind)
    shifted = torch.zeros(cols.numel() + 1, dtype=cols.dtype, device="cuda")[1:]
    shifted.copy_(cols)
    idx = np.nonzero((host[:-1] == ord("a")) & (host[1:] == ord("b")))[0]
    want = np.stack([idx, idx + 2], axis=1).astype(np.int64)
    for c in (cols, shifted):
        got, total = rx.matches(c, st, n, 5, k)
        assert total == len(want) and np.array_equal(got.cpu().numpy(), want)
    cap = len(want) // 2 + 1
    got, total = rx.matches(cols, st, n, 5, k, cap=cap)
    assert total == len(want) and np.array_equal(got.cpu().numpy(), want[:cap])


def test_span_longer_than_a_record(lib):
    """Group 1 spans the whole text: 2^21 - 2 bytes still fit a record, 2^21 - 1 do not."""
    rx = lib(W.AB_RE)
    for n in ((1 << 21) - 2, (1 << 21) - 1, (1 << 21) + 5):
        t = torch.from_numpy(W.ab_text(n, seed=3)).cuda()
        cols, st, k = rx.parse(t)
        got, total = rx.matches(cols, st, n, 1, k)
        assert total == 1 and got.cpu().numpy().tolist() == [[0, n]]
