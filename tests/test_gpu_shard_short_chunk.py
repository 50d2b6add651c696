"""Slices whose last chunk is one byte or little more: it speculates from the byte
after the slice, and where it has more slots than a lane holds a warp takes
it (the lane walk), whose slots already are at the chunk's end when it is one
byte long.  A slice's device maps against the oracle's run of Eq. reacher."""
import pytest

import workloads as W
from oracle import parallel_equations as pe
from oracle import speculation
from oracle.re_front import compile_re

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

AT = 64 * 50                                 # the slice's start in the text


@pytest.fixture(scope="module")
def log():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2503_06763_gb300 import Regex
    rx, c = Regex(W.LOG_RE), compile_re(W.LOG_RE)

    def as_set(v):
        return frozenset(q for q in range(c.ell) if (int(v[q >> 6]) >> (q & 63)) & 1)

    sets = [[as_set(rx.state_bits(fwd, s)) for s in range(rx.info["fwd_states" if fwd else "bwd_states"] + 1)]
            for fwd in (True, False)]
    host = W.log_text(20_000, seed=57)
    return rx, c, host, torch.from_numpy(host.copy()).cuda(), sets


# slices of one byte, and of one to five bytes more than one or two chunks of 256
@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 257, 258, 260, 261, 513])
def test_maps(log, n):
    rx, c, host, text, (fset, bset) = log
    nf, nb = rx.shard_map_size()
    m = speculation.Machine(c)
    fwd = {S: s for s, S in enumerate(fset)}
    bwd = {S: s for s, S in enumerate(bset)}
    starts = [a for a in range(AT, AT + 6400, 16)      # last chunks with more slots than a lane holds
              if len(speculation.backward_starts(m, int(host[a + n - 1]), int(host[a + n]), "me")) > 4]
    assert len(starts) >= 10
    for a in starts[:10]:
        b = a + n
        piece = host[a:b].tobytes()
        dev = rx.shard_map(text[a:b], True, True)
        edge_f = {pe.run(c, fset[s], host[a - 1:a].tobytes()) for s in range(nf)}
        edge_b = {pe.run(c, bset[s], host[b:b + 1].tobytes(), reverse=True) for s in range(nb)}
        for S in edge_f:
            assert fset[int(dev[fwd[S]])] == pe.run(c, S, piece), (a, sorted(S))
        for S in edge_b:
            assert bset[int(dev[nf + bwd[S]])] == pe.run(c, S, piece, reverse=True), (a, sorted(S))
