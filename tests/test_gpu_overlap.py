"""Calls queued back to back.  Decode steps, and every launch of a call but its first, may
start while the kernel before them still runs, so a chain in which each call reads what the
one before wrote (fields, states, coefficients, drive history) must give the same bits as
the chain with a device synchronisation after every call, and as its captured graph."""
import numpy as np
import pytest

import oracle
from synth import make_inputs, make_mixer_inputs
from tests._util import TOL, assert_close, to_dev, to_np

torch = pytest.importorskip("torch")
rlm = pytest.importorskip("paper_2607_05583_gb300")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    from paper_2607_05583_gb300 import build
    build.build()
    return rlm.load_library()


def _fields(L, D, M, dtype, K=4):
    inp = make_inputs(1, L, D, M, dtype, seed=L + M, with_dy=True)
    mx = make_mixer_inputs(inp, K, seed=M)
    return dict(p=rlm.Params.from_arrays(*inp.params()), x=to_dev(inp.x, dtype), dy=to_dev(inp.dy, dtype),
                g=to_dev(mx.g, dtype), local=rlm.Local.from_arrays(mx.conv_w, mx.scale),
                c_raw=np.random.default_rng(M).standard_normal((8, 8)), L=L, D=D, M=M, K=K)


def _buffers(f):
    e = lambda: torch.zeros_like(f["x"])
    t = lambda: torch.zeros_like(f["x"][0, :1])
    return dict(y=e(), dx=e(), s=rlm.State.empty(1, f["D"], f["M"]), gr=rlm.Grads.empty(f["D"], f["M"]),
                conv=rlm.ConvState.empty(1, f["D"], f["K"], dtype=f["x"].dtype), a=t(), b=t(),
                ws=torch.empty(64 << 20, dtype=torch.uint8, device="cuda"))


# Each chain yields after every call.
def _scan_decode(f, o):
    rlm.rlm_mix_prefill(f["x"], f["p"], o["y"], o["s"], workspace=o["ws"])
    yield
    rlm.rlm_mix_decode(o["y"][0, -1:], o["s"], o["a"])   # the layer above takes the last output
    yield
    rlm.rlm_mix_decode(o["a"], o["s"], o["b"])
    yield


def _mixer_decode(f, o):
    c = rlm.Coupling(f["cr"], 0.5)
    rlm.rlm_mixer_prefill(f["x"], f["g"], f["p"], f["local"], o["y"], state_out=o["s"], conv_out=o["conv"],
                          workspace=o["ws"], coupling=c)
    yield
    rlm.rlm_mixer_decode(o["y"][0, -1:], f["g"][0, -1:], o["s"], f["local"], o["conv"], o["a"], coupling=c)
    yield
    rlm.rlm_mixer_decode(o["a"], f["g"][0, :1], o["s"], f["local"], o["conv"], o["b"], coupling=c)
    yield


def _backward_decode(f, o):
    rlm.rlm_state_init(o["s"], f["p"])
    yield
    rlm.rlm_mix_decode(f["x"][0, :1], o["s"], o["a"])
    yield
    rlm.rlm_mix_backward(f["dy"], f["x"], f["p"], o["dx"], o["gr"], workspace=o["ws"])
    yield
    rlm.rlm_mix_decode(o["dx"][0, -1:], o["s"], o["b"])
    yield
    rlm.rlm_mix_prefill(o["dx"], f["p"], o["y"], None, workspace=o["ws"])
    yield


def _results(o):
    return [t.clone() for t in (o["y"], o["dx"], o["s"].s, o["conv"].u, o["a"], o["b"], o["gr"].decay, o["gr"].freq,
                                o["gr"].amp, o["gr"].phase)]


@pytest.mark.parametrize("chain", [_scan_decode, _mixer_decode, _backward_decode])
@pytest.mark.parametrize("L,D,M,dtype", [(5000, 64, 20, "f32"), (3000, 256, 16, "bf16"), (2500, 128, 32, "bf16"),
                                         (700, 64, 33, "bf16")])
def test_a_queued_chain_equals_the_synchronised_one(chain, L, D, M, dtype):
    f = _fields(L, D, M, dtype)
    f["cr"] = torch.from_numpy(f["c_raw"].astype(np.float32)).cuda()
    zero = lambda o: [t.zero_() for t in (o["y"], o["dx"], o["s"].s, o["s"].coef, o["conv"].u, o["a"], o["b"],
                                          o["gr"].decay, o["gr"].freq, o["gr"].amp, o["gr"].phase)]
    o = _buffers(f)
    zero(o)
    for _ in chain(f, o):
        torch.cuda.synchronize()
    want = _results(o)
    for _ in range(3):
        zero(o)
        for _ in chain(f, o):
            pass
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(want, _results(o)))
    graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        graph.capture_begin()
        for _ in chain(f, o):
            pass
        graph.capture_end()
    torch.cuda.current_stream().wait_stream(side)
    for _ in range(2):
        zero(o)
        graph.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(want, _results(o)))


# The coupling matrix is written by the kernel right before every step: matrices of fewer and
# of more entries than a block has threads (256 with several blocks a row, 512 with one).
@pytest.mark.parametrize("B,D,M,H,dtype", [(2, 256, 16, 16, "bf16"), (3, 240, 16, 20, "f32"), (2, 128, 32, 64, "f32"),
                                           (80, 256, 16, 32, "bf16"), (90, 384, 8, 24, "f32"), (2, 408, 4, 51, "f32")])
def test_coupled_steps_take_the_matrix_written_just_before(B, D, M, H, dtype):
    T, K = 3, 2
    inp = make_inputs(B, T, D, M, dtype, seed=B + H)
    mx = make_mixer_inputs(inp, K, seed=H)
    c_np = np.random.default_rng(H).standard_normal((H, H))
    want = torch.from_numpy(c_np.astype(np.float32)).cuda()
    c = rlm.Coupling(torch.empty_like(want), 0.5)
    x, g = to_dev(inp.x, dtype), to_dev(mx.g, dtype)
    tokens = [(x[:, t].contiguous(), g[:, t].contiguous()) for t in range(T)]
    st, local = rlm.State.empty(B, D, M), rlm.Local.from_arrays(mx.conv_w, mx.scale)
    rlm.rlm_state_init(st, rlm.Params.from_arrays(*inp.params()))
    conv, z = rlm.ConvState(to_dev(mx.conv_in, dtype)), torch.empty(T, B, D, dtype=x.dtype, device="cuda")
    for t, (xt, gt) in enumerate(tokens):
        c.c_raw.fill_(9.0 + t)
        c.c_raw.copy_(want)
        rlm.rlm_mixer_decode(xt, gt, st, local, conv, z[t], coupling=c)
        c.c_raw.fill_(-5.0)
    torch.cuda.synchronize()
    ref = oracle.mixer_prefill(inp.x, mx.g, *inp.params(), mx.conv_w, mx.scale, conv_in=mx.conv_in,
                               coupling=(c_np, 0.5))[0]
    assert_close(to_np(z.transpose(0, 1)), ref, TOL[dtype], "z")


# A call on another stream than the current one, without a workspace: its workspace is neither
# a block that work of the current stream still uses, nor given to that stream while the call runs.
@pytest.mark.parametrize("native", [True, False])
@pytest.mark.parametrize("handle", [False, True])
@pytest.mark.parametrize("B,L,D,M,dtype", [(1, 9000, 64, 20, "f32"), (2, 2000, 128, 32, "bf16")])
def test_workspace_of_a_call_on_a_side_stream(monkeypatch, native, handle, B, L, D, M, dtype):
    if not native:
        monkeypatch.setattr(rlm, "_native", _NoNative())
    inp = make_inputs(B, L, D, M, dtype, seed=L, with_dy=True)
    p, x, dy = rlm.Params.from_arrays(*inp.params()), to_dev(inp.x, dtype), to_dev(inp.dy, dtype)
    need = rlm.rlm_prefill_workspace_size(B, L, D, M, x.dtype), rlm.rlm_backward_workspace_size(B, L, D, M, x.dtype)
    assert min(need) > 0

    def calls(stream, y, dx, gr):
        rlm.rlm_mix_prefill(x, p, y, stream=stream)
        rlm.rlm_mix_backward(dy, x, p, dx, gr, stream=stream)

    outs = [(torch.zeros_like(x), torch.zeros_like(x), rlm.Grads.empty(D, M)) for _ in range(2)]
    calls(None, *outs[0])
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    for n in need:   # blocks of these sizes are free, and the current stream still writes them
        block = torch.empty(n, dtype=torch.uint8, device="cuda")
        torch.cuda._sleep(2_000_000)
        block.fill_(0x7f)
        del block
    with torch.cuda.stream(side):
        torch.cuda._sleep(1_000_000)   # the current stream's later work runs first
    calls(side.cuda_stream if handle else side, *outs[1])
    for n in need:
        torch.empty(n, dtype=torch.uint8, device="cuda").fill_(0x7f)
    torch.cuda.synchronize()
    for a, b in zip(outs[0][:2], outs[1][:2]):
        assert torch.equal(a, b)
    for k in ("decay", "freq", "amp", "phase"):
        assert torch.equal(getattr(outs[0][2], k), getattr(outs[1][2], k))


class _NoNative:
    """Hands every call to the ctypes route."""
    def __getattr__(self, name):
        return lambda *args: None


@pytest.mark.parametrize("native", [True, False])
def test_default_stream_by_handle_while_another_is_current(monkeypatch, native):
    if not native:
        monkeypatch.setattr(rlm, "_native", _NoNative())
    inp = make_inputs(1, 5000, 64, 20, "f32", seed=1)
    p, x = rlm.Params.from_arrays(*inp.params()), to_dev(inp.x, "f32")
    want, y = torch.zeros_like(x), torch.zeros_like(x)
    rlm.rlm_mix_prefill(x, p, want)
    torch.cuda.synchronize()
    with torch.cuda.stream(torch.cuda.Stream()):
        for h in (0, 1):
            y.zero_()
            torch.cuda.synchronize()
            rlm.rlm_mix_prefill(x, p, y, stream=h)
            torch.cuda.synchronize()
            assert torch.equal(y, want)
