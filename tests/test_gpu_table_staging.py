"""Tables copied into shared memory before a walk: automata whose table and
column-dictionary sizes leave remainders of a block's copy (eight entries of a
thread, 16-byte vectors), at texts around a 64-column group, against the oracle."""
import numpy as np
import pytest

import workloads as W
from oracle import serial
from oracle.re_front import compile_re

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def lib():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2503_06763_gb300 import Regex
    return Regex


@pytest.mark.parametrize("kind", ["dict", "dense"])
@pytest.mark.parametrize("k", [1, 4, 7, 9, 11])
def test_suffix_family(lib, k, kind):
    pattern = "(a|b)*a" + "(a|b)" * k
    rx = lib(pattern)
    front = compile_re(pattern)
    for n in (k + 1, 63, 64, 65, 191, 4097):
        host = W.ab_text(n, seed=n)[:n].copy()
        host[n - 1 - k] = ord("a")                   # accepted
        ids, table = serial.parse_ids(front, host)
        want = table[ids]
        t = torch.from_numpy(host).cuda()
        for shape in (2, 4):
            cols, st, got_kind = rx.parse(t, chunk_len=64, reach_shape=shape, kind=kind)
            assert int(st.item()) == 0
            assert np.array_equal(rx.decode(cols.cpu().numpy(), got_kind), want), (n, shape)
