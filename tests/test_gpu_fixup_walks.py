"""The fix-up of checkpoints where a chunk's runs stay apart past what it records:
32 boundaries of 64 bytes, fewer with many runs.  Chunks of just that length,
one boundary more and much more, every item of a block with a walk or some of
them, ragged last chunks, single texts and batches.  Against the oracle."""
import numpy as np
import pytest

from oracle import serial
from oracle.re_front import compile_re

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _same(n):
    return np.full(n, ord("a"), dtype=np.uint8)


def _some(n):
    x = _same(n)                                       # runs meet at a b: one every 3 to 30 thousand letters
    at = np.cumsum(2 * np.random.default_rng(n).integers(1500, 15_000, n // 3000 + 2) + 1) - 1
    x[at[at < n]] = ord("b")
    x[n - 1] = ord("b")
    return x


CASES = {"aa": ("(aa)*", _same), "six": ("(aaaaaa)*", _same), "twelve": ("(aaaaaaaaaaaa)*", _same),
         "some": ("((aa)*(b|c))*", _some)}


@pytest.fixture(scope="module")
def lib():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2503_06763_gb300 import Batch, Regex
    return Batch, Regex


@pytest.mark.parametrize("name", sorted(CASES))
@pytest.mark.parametrize("k", [512, 576, 1024, 1088, 2048, 2112, 2176, 4096])
def test_columns(lib, name, k):
    Batch, Regex = lib
    pattern, make = CASES[name]
    rx, c = Regex(pattern), compile_re(pattern)
    hosts = [make(12 * (q * k // 12) + 12 * e) for q, e in ((1, 0), (3, 1), (40, 3), (70, 171))]
    texts = [torch.from_numpy(h).cuda() for h in hosts]
    outs, status, kinds = Batch([rx] * len(hosts), [h.size for h in hosts], chunk_len=k).parse(texts)
    for j, (host, t) in enumerate(zip(hosts, texts)):
        ids, table = serial.parse_ids(c, host)
        want = table[ids]
        code = 0 if serial.accepted(want) else 1
        for shape in (2, 3, 4):
            cols, st, kind = rx.parse(t, chunk_len=k, reach_shape=shape)
            assert int(st.item()) == code, (host.size, shape)
            assert np.array_equal(rx.decode(cols.cpu().numpy(), kind), want), (host.size, shape)
        assert int(status[j].item()) == code
        assert np.array_equal(rx.decode(outs[j].cpu().numpy(), kinds[j]), want), host.size
