"""The join's scan over units of one, four and eight chunks: chunk counts around
those where the unit changes and where the last unit is partial, runs that
never meet, that meet in some chunks, accepted and rejected texts, with columns
and recognized, by warp pairs and by the lane walk.  Against the oracle."""
import numpy as np
import pytest

import workloads as W
from oracle import serial
from oracle.re_front import compile_re

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

CHUNKS = [2, 8191, 8192, 8193, 8195, 8196, 8197, 32_767, 32_768, 32_769, 32_775, 32_776]
CASES = {
    "aa": ("(aa)*", lambda n: np.full(n, ord("a"), dtype=np.uint8)),
    "six": ("(aaaaaa)*", lambda n: np.full(n, ord("a"), dtype=np.uint8)),
    # runs meet at a b: one every 700 to 7000 letters
    "some": ("((aa)*(b|c))*", lambda n: _some(n)),
    "dna": (W.DNA_RE, lambda n: W.dna_text(n, seed=n, mean_gap=1000)),
}


def _some(n):
    x = np.full(n, ord("a"), dtype=np.uint8)
    at = np.cumsum(2 * np.random.default_rng(n).integers(350, 3500, n // 700 + 2) + 1) - 1
    x[at[at < n]] = ord("b")
    x[n - 1] = ord("b")
    return x


@pytest.fixture(scope="module")
def lib():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2503_06763_gb300 import Regex
    return Regex


@pytest.mark.parametrize("name", sorted(CASES))
@pytest.mark.parametrize("c", CHUNKS)
def test_units(lib, name, c):
    pattern, make = CASES[name]
    rx, oracle = lib(pattern), compile_re(pattern)
    for n in (64 * (c - 1) + 2, 64 * c):
        host = make(n)
        for spoil in (None, n // 3):
            if spoil is not None:
                host = host.copy()
                host[spoil] = ord("x")
            ids, table = serial.parse_ids(oracle, host)
            want = table[ids]
            status = 0 if serial.accepted(want) else 1
            t = torch.from_numpy(host).cuda()
            for shape in (1, 2):
                cols, st, kind = rx.parse(t, chunk_len=64, reach_shape=shape)
                _, rst, _ = rx.parse(t, chunk_len=64, reach_shape=shape, recognize_only=True)
                torch.cuda.synchronize()
                assert int(st.item()) == int(rst.item()) == status, (n, spoil, shape)
                assert np.array_equal(rx.decode(cols.cpu().numpy(), kind), want), (n, spoil, shape)
