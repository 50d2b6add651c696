"""The rebuild's routes: short pieces by the thread where there are many of them,
tables read where they are or staged by their rows and the text's length.  The
columns must be the ones archived, on both sides of each line."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def native():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2503_06763_gb300 import native
    return native


def _round_trip(native, n, n_ids, K, cb, shift=0):
    rng = np.random.default_rng(n + n_ids)
    text = rng.integers(97, 101, n).astype(np.uint8)
    cols = np.zeros(n + 1, dtype={1: np.uint8, 2: np.uint16}[cb])
    cols[1:] = np.where(rng.random(n) < 0.05, rng.integers(0, n_ids, n), (text.astype(np.int64) * 7) % n_ids)
    cols[n // 2] = n_ids - 1
    buf = torch.zeros(n + 64, dtype=torch.uint8, device="cuda")
    d_text = buf[shift:shift + n]
    d_text.copy_(torch.from_numpy(text))
    got, st = native.slpf_dfa_decode(native.slpf_dfa_encode(cols, text, K), d_text, cb)
    assert int(st.item()) == 0
    assert np.array_equal(got.cpu().numpy().view(cols.dtype), cols)


# 64 K pieces and one more; an interval that is no multiple of 16 and a text that is not aligned
@pytest.mark.parametrize("K", [256, 272, 300, 496, 512])
@pytest.mark.parametrize("more", [-1, 0, 1])
def test_many_pieces(native, K, more):
    for shift in (0, 3):
        _round_trip(native, (64 * K - 1) * K + more, 100, K, 1, shift)


@pytest.mark.parametrize("n_ids", [192, 193, 254, 255, 256, 400, 401])
def test_rows(native, n_ids):
    _round_trip(native, 50_001, n_ids, 1000, 2)


@pytest.mark.parametrize("less", [0, 1])
def test_rows_of_a_long_text(native, less):
    _round_trip(native, 193 * 65536 - less, 193, 4096, 2)
