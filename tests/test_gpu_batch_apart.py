"""Batches under automata whose speculative runs can stay apart for a whole text,
so that chunks are evaluated after one another: small tables (warp pairs) and
large ones (the lane walk), two runs and more than a lane holds, short texts
and one of many chunks, accepted and rejected, with columns and recognized.
Short texts against the oracle, all of them against the single parse by warp
pairs on 256-byte chunks."""
import numpy as np
import pytest

import workloads as W
from oracle import serial
from oracle.re_front import compile_re

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

TWENTY = "abcdefghijklmnopqrst"


def _same(n, seed):
    return np.full(n, ord("a"), dtype=np.uint8)


def _blocks(width):
    def make(n, seed):                                     # letters in blocks: some runs meet at block ends
        return np.repeat(np.random.default_rng(seed).integers(97, 117, n // width + 1).astype(np.uint8), width)[:n].copy()
    return make


CASES = {
    "aa": ("(aa)*", _same),
    "six": ("(aaaaaa)*", _same),
    "last": ("(a*b)*c|(b*a)*d", lambda n, seed: np.concatenate([W.ab_text(n, seed=seed)[:max(n - 2, 0)],
                                                                np.frombuffer(b"bc", np.uint8)[:n]])),
    "dna": (W.DNA_RE, lambda n, seed: W.dna_text(n, seed=seed, mean_gap=2000)),
    "twos-same": ("(" + "|".join(c * 2 for c in TWENTY) + ")*", _same),
    "twos": ("(" + "|".join(c * 2 for c in TWENTY) + ")*", _blocks(2)),
    "sixes-same": ("(" + "|".join(c * 6 for c in TWENTY) + ")*", _same),
    "sixes": ("(" + "|".join(c * 6 for c in TWENTY) + ")*", _blocks(6)),
    "log-one-line": (W.LOG_RE, lambda n, seed: np.concatenate([_same(n - 1, seed), np.frombuffer(b"\n", np.uint8)])),
}
SIZES = (1, 6, 63, 65, 257, 600, 4098, 8193, 66_000, 1_500_006)


@pytest.fixture(scope="module")
def lib():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2503_06763_gb300 import Batch, Regex
    return Batch, Regex


@pytest.mark.parametrize("chunk_len", [0, 64, 192])
@pytest.mark.parametrize("name", sorted(CASES))
def test_batch(lib, name, chunk_len):
    Batch, Regex = lib
    pattern, make = CASES[name]
    rx, c = Regex(pattern), compile_re(pattern)
    hosts = [make(n, n) for n in SIZES if n < 100_000 or chunk_len == 0]
    spoiled = hosts[6].copy()
    spoiled[-3] = 0x01
    hosts.append(spoiled)
    texts = [torch.from_numpy(h).cuda() for h in hosts]
    want = [rx.parse(t, chunk_len=256, reach_shape=2) for t in texts]
    b = Batch([rx] * len(hosts), [h.size for h in hosts], chunk_len=chunk_len)
    outs, status, kinds = b.parse(texts)
    r = Batch([rx] * len(hosts), [h.size for h in hosts], chunk_len=chunk_len, recognize_only=True)
    _, rstatus, _ = r.parse(texts)
    torch.cuda.synchronize()
    for j, h in enumerate(hosts):
        cols, st, _ = want[j]
        assert int(status[j].item()) == int(rstatus[j].item()) == int(st.item()), (j, h.size)
        assert torch.equal(outs[j], cols), (j, h.size)
        if h.size < 10_000:
            ids, table = serial.parse_ids(c, h)
            exact = table[ids]
            assert int(st.item()) == (0 if serial.accepted(exact) else 1), (j, h.size)
            assert np.array_equal(rx.decode(outs[j].cpu().numpy(), kinds[j]), exact), (j, h.size)


@pytest.mark.parametrize("recognize", [False, True])
@pytest.mark.parametrize("more", [0, 1])
def test_groups_beside_a_lane_walk(lib, more, recognize):
    """Groups of small tables beside one that takes the lane walk, each of 1 MiB
    in all (they join it) or of a byte more (they do not), in texts of many sizes."""
    Batch, Regex = lib
    log = W.log_text(300_000, seed=5)
    items = [("log", W.LOG_RE, log), ("log", W.LOG_RE, log[:1].copy())]
    for name in ("aa", "six", "dna"):
        pattern, make = CASES[name]
        sizes = [7, 600, 8194, 66_000, 280_000]
        sizes.append((1 << 20) + more - sum(sizes))
        items += [(name, pattern, make(n, n)) for n in sizes]
    rxs = {name: Regex(pattern) for name, pattern, _ in items}
    texts = [torch.from_numpy(h).cuda() for _, _, h in items]
    b = Batch([rxs[name] for name, _, _ in items], [h.size for _, _, h in items], recognize_only=recognize)
    outs, status, _ = b.parse(texts)
    torch.cuda.synchronize()
    for j, (name, _, h) in enumerate(items):
        cols, st, _ = rxs[name].parse(texts[j], chunk_len=256, reach_shape=2)
        assert int(status[j].item()) == int(st.item()), (name, h.size)
        assert recognize or torch.equal(outs[j], cols), (name, h.size)
