"""The lane walk (reach shape 1: speculative heads, then one run per chunk and
direction on through the next chunk's head) against the oracle, every column,
where it can go wrong: texts that end inside, on and after a 32-byte unit, a
64-byte chunk and a 32-chunk tile; chunks whose runs never meet, so that the
join evaluates them and walks the heads after them; more slots than a lane
holds; text buffers that are 16-byte but not 32-byte aligned; rejected texts."""
import numpy as np
import pytest

import workloads as W
from oracle import serial
from oracle.re_front import compile_re

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

# name, pattern, text of n bytes
CASES = {
    "aa": ("(aa)*", lambda n: np.full(n, ord("a"), dtype=np.uint8)),            # runs never meet
    "mixed": ("((aa)*b|c)*", lambda n: np.frombuffer((b"aab" + b"a" * 200 + b"bccaaaab") * (n // 211 + 1),
                                                      dtype=np.uint8)[:n].copy()),   # some meet late
    "dna": (W.DNA_RE, lambda n: W.dna_text(n, seed=n, mean_gap=300)),
    "ab": (W.AB_RE, lambda n: W.ab_text(n, seed=n)),
    "log": (W.LOG_RE, None),
}
LOG = W.log_text(90_000, seed=8)


@pytest.fixture(scope="module")
def lib():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2503_06763_gb300 import Regex
    return Regex


@pytest.mark.parametrize("name", sorted(CASES))
@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 63, 64, 65, 97, 64 * 32 - 1, 64 * 32, 64 * 33 + 5, 64 * 64 + 32, 70_001])
def test_every_column(lib, name, n):
    pattern, make = CASES[name]
    host = LOG[:n].copy() if make is None else make(n)
    rx = lib(pattern)
    ids, table = serial.parse_ids(compile_re(pattern), host)
    want = table[ids]
    status = 0 if serial.accepted(want) else 1
    buf = torch.zeros(n + 64, dtype=torch.uint8, device="cuda")
    for chunk_len, shift in ((64, 0), (64, 16), (192, 0), (0, 16)):
        t = buf[shift:shift + n]
        t.copy_(torch.from_numpy(host))
        cols, st, kind = rx.parse(t, chunk_len=chunk_len, reach_shape=1)
        _, rst, _ = rx.parse(t, chunk_len=chunk_len, reach_shape=1, recognize_only=True)
        torch.cuda.synchronize()
        assert int(st.item()) == int(rst.item()) == status, (chunk_len, shift)
        got = rx.decode(cols.cpu().numpy(), kind)
        bad = np.nonzero(np.any(got != want, axis=1))[0]
        assert bad.size == 0, (chunk_len, shift, bad[:5].tolist())
