"""A damaged archive whose table names an id that is none of its own: the
rebuild reports it, whatever the interval, the width of the ids and where the
table is read from.  The damaged entry is the one that the most columns take."""
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


def _columns(name, native):
    if name == "log":                                     # one-byte ids, the table staged
        text = W.log_text(60_000, seed=6)
        cols, _, _ = native.Regex(W.LOG_RE).parse(torch.from_numpy(text.copy()).cuda())
        return text, cols.cpu().numpy().view(np.uint8)
    rng = np.random.default_rng(3)                        # more ids than a byte; the largest table is not staged
    text = rng.integers(97, 101, 60_000).astype(np.uint8)
    cols = np.zeros(text.size + 1, dtype=np.uint16)
    cols[1:] = np.where(rng.random(text.size) < 0.05, rng.integers(0, int(name), text.size), text - 96)
    cols[50] = int(name) - 1
    return text, cols


@pytest.mark.parametrize("name", ["log", "300", "20000"])
@pytest.mark.parametrize("K", [64, 255, 256, 4096, 65_536])
def test_flagged(native, name, K):
    text, cols = _columns(name, native)
    d_text, cb = torch.from_numpy(text.copy()).cuda(), cols.dtype.itemsize
    arch = native.slpf_dfa_encode(cols, text, K)
    n_ids = int(cols.max()) + 1
    table = arch[48:48 + n_ids * 512].view(np.uint16).reshape(n_ids, 256)
    took = table[cols[:-1], text] == cols[1:]
    pairs, uses = np.unique(cols[:-1][took].astype(np.int64) * 256 + text[took], return_counts=True)
    v, a = divmod(int(pairs[np.argmax(uses)]), 256)
    right = int(table[v, a])
    for wrong in (n_ids, 256 + right, 0xFFFE):
        if wrong < n_ids:
            continue
        table[v, a] = wrong
        _, st = native.slpf_dfa_decode(arch, d_text, cb)
        assert int(st.item()) == -9, wrong
    table[v, a] = right
    got, st = native.slpf_dfa_decode(arch, d_text, cb)
    assert int(st.item()) == 0
    assert np.array_equal(got.cpu().numpy().view(cols.dtype), cols)
