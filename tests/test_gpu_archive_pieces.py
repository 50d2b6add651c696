"""The archive rebuild with a warp per piece (intervals of 256 columns and
more): pieces of whole and part windows of 4096 columns, pieces longer than a
window, more exceptions than are staged and none at all, ids of one and two
bytes, unaligned text; the rebuilt columns must be the parse's."""
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


TEXTS = {
    "log": (W.LOG_RE, lambda n: W.log_text(n, seed=4)),
    "dna": (W.DNA_RE, lambda n: W.dna_text(n, seed=4)),
    "ab": (W.AB_RE, lambda n: W.ab_text(n, seed=4)),
    "no-exceptions": ("(a|b)*", lambda n: np.full(n, ord("a"), dtype=np.uint8)),
}


@pytest.mark.parametrize("name", sorted(TEXTS))
@pytest.mark.parametrize("K", [255, 256, 257, 1000, 4095, 4096, 4097, 10_000, 65_536])
def test_pieces(native, name, K):
    pattern, make = TEXTS[name]
    rx = native.Regex(pattern)
    for n in (0, 1, 255, 256, 4096, 8191, 70_003):
        host = make(n) if n else np.zeros(0, dtype=np.uint8)
        buf = torch.zeros(host.size + 64, dtype=torch.uint8, device="cuda")
        for shift in (0, 3):
            text = buf[shift:shift + host.size]
            text.copy_(torch.from_numpy(host))
            cols, st, _ = rx.parse(text.clone())
            cb = cols.element_size()
            arch = native.slpf_dfa_encode(cols.cpu().numpy().view({1: np.uint8, 2: np.uint16}[cb]), host.tobytes(), K)
            got, status = native.slpf_dfa_decode(arch, text, cb)
            torch.cuda.synchronize()
            assert int(status.item()) == 0
            assert torch.equal(got.view(torch.uint8), cols.view(torch.uint8)), (n, shift)
            if cb == 1 or n > 9000:
                continue
            wide = native.slpf_dfa_decode(arch, text, 4)[0]        # the same ids in wider columns
            assert torch.equal(wide, cols.view(torch.int16).to(torch.int32)), (n, shift)
