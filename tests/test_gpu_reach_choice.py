"""The built-in choice of reach shape and chunk length against warp pairs on
256-byte chunks: automata whose runs always meet and ones whose runs can stay
apart for ever, small and large, at lengths around those where the chunk length
moves; and a workspace that holds only the plain layout."""
import ctypes

import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

# name, pattern, letters
CASES = {
    "ab": (W.AB_RE, "ab"),                                                   # every pair meets
    "suffix3": ("(a|b)*a(a|b)(a|b)(a|b)", "ab"),
    "suffix8": ("(a|b)*a" + "(a|b)" * 8, "ab"),                              # more states than a byte
    "aa": ("(aa)*", "a"),                                                    # runs never meet
    "parity": ("((a|b)(a|b))*a?", "ab"),
    "last": ("(a*b)*c|(b*a)*d", "ab"),                                       # meet on one letter only
    "dna": (W.DNA_RE, "ACGT"),
}


@pytest.fixture(scope="module")
def native():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2503_06763_gb300 import native
    return native


@pytest.mark.parametrize("name", sorted(CASES))
@pytest.mark.parametrize("n", [1, 64, 255, 256, 257, 524_287, 524_289, 1_048_577, 2_000_003])
def test_same_columns(native, name, n):
    pattern, letters = CASES[name]
    rx = native.Regex(pattern)
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    pick = torch.randint(0, len(letters), (n,), generator=g, device="cuda")
    t = torch.tensor([ord(c) for c in letters], dtype=torch.uint8, device="cuda")[pick]
    for last in (None, "c", "?"):
        if last:
            t[n - 1] = ord(last)
        want, wst, _ = rx.parse(t, chunk_len=256, reach_shape=2)
        got, st, _ = rx.parse(t)
        _, rst, _ = rx.parse(t, recognize_only=True)
        torch.cuda.synchronize()
        assert int(wst.item()) == int(st.item()) == int(rst.item()), last
        assert torch.equal(got, want), last


@pytest.mark.parametrize("recognize", [False, True])
def test_workspace_of_the_plain_layout(native, recognize):
    """The rule wants 320-byte chunks for a recognizer of 20 MB; a workspace
    that holds 384-byte chunks is taken, one that does not is refused."""
    rx = native.Regex(W.LOG_RE)
    line = torch.from_numpy(W.log_text(50_000, seed=2).copy()).cuda()
    t = line.repeat(20_000_000 // line.numel())              # whole lines
    n = t.numel()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    plain = max(256, -(-(-(-n // (sms * 384))) // 64) * 64)
    flags = native.RE_PARSE_RECOGNIZE_ONLY if recognize else 0
    want, wst, kind = rx.parse(t, chunk_len=plain, recognize_only=recognize)
    _, cb, _ = rx.layout(n, "auto")
    size = rx.workspace_size(n, plain, flags)
    assert rx.workspace_size(n, 0, flags) >= size
    lib = native.load()
    for room, expect in ((size, 0), (size - 256, -8)):
        ws = torch.empty(room, dtype=torch.uint8, device="cuda")
        out = torch.zeros_like(want) if want is not None else None
        st = torch.full((1,), 7, dtype=torch.int32, device="cuda")
        slpf = native.Slpf(native.KINDS[kind], cb, 0, out.data_ptr() if out is not None else None,
                           out.numel() * out.element_size() if out is not None else 0, st.data_ptr())
        opts = native.ParseOpts(native.KINDS[kind], 0, flags, 0, None)
        rc = lib.re_parse(rx._h, t.data_ptr(), n, ctypes.c_void_p(torch.cuda.current_stream().cuda_stream),
                          ctypes.byref(slpf), ws.data_ptr(), ws.numel(), ctypes.byref(opts))
        torch.cuda.synchronize()
        assert rc == expect
        if rc == 0:
            assert int(st.item()) == int(wst.item())
            assert out is None or torch.equal(out, want)
