"""A batch's workspace against the sum of its texts' own: each text's chunks are
no shorter than its group alone would get (the group's bytes over 384 chunks a
multiprocessor, at least 32 chunks a text where it can), and beside the texts'
workspaces there are only descriptors, so a workspace of that sum and of the
descriptors' part (three tensor maps, the parameters and the place in the prefix sums) holds a batch
whatever its shape."""
import ctypes

import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

APART = "(" + "|".join(c * 2 for c in "abcdefghijklmnopqrst") + ")*"     # large tables, runs that can stay apart


@pytest.fixture(scope="module")
def native():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2503_06763_gb300 import native
    return native


def _up(v, step):
    return -(-v // step) * step


SHAPES = {
    "one-byte": [1], "tiny": [5] * 3, "empty": [0, 0], "chunk": [256], "chunks": [257, 8192, 8193],
    "short": [4080] * 256, "ragged": [1 << q for q in range(23)], "long": [64 << 20], "four": [16 << 20] * 4,
}


@pytest.mark.parametrize("recognize", [False, True])
@pytest.mark.parametrize("pattern", [W.LOG_RE, W.AB_RE, W.DNA_RE, "(aa)*", APART, "(a|b)*a" + "(a|b)" * 9])
@pytest.mark.parametrize("shape", sorted(SHAPES))
def test_sum_of_texts(native, pattern, shape, recognize):
    rx, lens = native.Regex(pattern), SHAPES[shape]
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    flags = native.RE_PARSE_RECOGNIZE_ONLY if recognize else 0
    group = max(256, _up(-(-sum(lens) // (sms * 384)), 64))
    room = 0
    for n in lens:
        k = max(256, min(group, _up(-(-n // 32), 64)))
        room += (_up(rx.workspace_size(n, k, flags), 256) if n else 0) + 3 * 128 + 768
    b = native.Batch([rx] * len(lens), lens, recognize_only=recognize)
    size = ctypes.c_uint64()
    native.check(native.load().re_batch_workspace_size(b._b, ctypes.byref(size)))
    assert size.value <= room + 5 * 256                           # rounding of the descriptors
