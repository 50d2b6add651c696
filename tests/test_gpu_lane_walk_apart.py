"""The lane walk where a chunk has more slots than a lane keeps runs and they stay
apart: to the chunk's end within what a warp walks, and past it, in one and in
two passes of eight slots; with columns, recognized, and as slices of a text.
Against the oracle."""
import numpy as np
import pytest

import workloads as W
from oracle import serial
from oracle.re_front import compile_re

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

TWENTY = "abcdefghijklmnopqrst"
CASES = {
    "six": "(aaaaaa)*",                                    # 6 slots each way
    "twelve": "(aaaaaaaaaaaa)*",                           # 12
    "seven-or-b": "((aaaaaaa)*(b|c))*",                    # some runs meet at a b
    "sixes": "(" + "|".join(c * 6 for c in TWENTY) + ")*",
}


def _texts(n):
    a = np.full(n, ord("a"), dtype=np.uint8)
    few = a.copy()
    few[(n // 7 // 2) * 7::501] = ord("b")
    return [a, few]


@pytest.fixture(scope="module")
def lib():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2503_06763_gb300 import Regex, shard
    return Regex, shard


@pytest.mark.parametrize("name", sorted(CASES))
@pytest.mark.parametrize("n", [1, 5, 12, 64, 65, 84, 192, 257, 504, 4096, 4098, 20_160, 70_001, 84_000])
def test_columns_and_verdict(lib, name, n):
    Regex, shard = lib
    rx, c = Regex(CASES[name]), compile_re(CASES[name])
    for host in _texts(n):
        ids, table = serial.parse_ids(c, host)
        want = table[ids]
        status = 0 if serial.accepted(want) else 1
        t = torch.from_numpy(host).cuda()
        for k in (64, 128, 192, 0):
            cols, st, kind = rx.parse(t, chunk_len=k, reach_shape=1)
            _, rst, _ = rx.parse(t, chunk_len=k, reach_shape=1, recognize_only=True)
            torch.cuda.synchronize()
            assert int(st.item()) == int(rst.item()) == status, k
            assert np.array_equal(rx.decode(cols.cpu().numpy(), kind), want), k


@pytest.mark.parametrize("name", sorted(CASES))
@pytest.mark.parametrize("n", [504, 4098, 20_160])
def test_slices(lib, name, n):
    Regex, shard = lib
    rx, c = Regex(CASES[name]), compile_re(CASES[name])
    for host in _texts(n):
        ids, table = serial.parse_ids(c, host)
        want = table[ids]
        for parts in (2, 3):
            cols, stats, accepted = shard.parse_in_slices(rx, torch.from_numpy(host).cuda(), parts)
            torch.cuda.synchronize()
            assert accepted == serial.accepted(want)
            assert (stats.cpu().numpy() == (0 if accepted else 1)).all()
            assert np.array_equal(rx.decode(cols.cpu().numpy(), rx.layout(1)[0]), want), parts


@pytest.mark.parametrize("k", [256, 576, 1024, 4096])
@pytest.mark.parametrize("n", [4095, 70_001, 200_003])
def test_runs_that_meet_late(lib, n, k):
    """The genome RE has up to eight runs for some hundred bytes: they meet in a
    lane's share of the chunk, down to few enough for the rest or to its end."""
    Regex, _ = lib
    rx, c = Regex(W.DNA_RE), compile_re(W.DNA_RE)
    host = W.dna_text(n, seed=n + k, mean_gap=700)
    for spoil in (None, n - 60):
        if spoil is not None:
            host[spoil] = ord("N")
        ids, table = serial.parse_ids(c, host)
        want = table[ids]
        t = torch.from_numpy(host).cuda()
        cols, st, kind = rx.parse(t, chunk_len=k, reach_shape=1)
        _, rst, _ = rx.parse(t, chunk_len=k, reach_shape=1, recognize_only=True)
        torch.cuda.synchronize()
        assert int(st.item()) == int(rst.item()) == (0 if serial.accepted(want) else 1)
        assert np.array_equal(rx.decode(cols.cpu().numpy(), kind), want)
