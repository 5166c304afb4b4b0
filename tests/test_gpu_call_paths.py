"""The two call paths of the binding (native, and ctypes where that is not built) make the
same calls: all five entry points, with and without their optional arguments, bit by bit."""
import numpy as np
import pytest

from synth import make_inputs, make_mixer_inputs
from tests._util import to_dev

torch = pytest.importorskip("torch")
rlm = pytest.importorskip("paper_2607_05583_gb300")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("full", [True, False])
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_native_and_ctypes_calls_agree(monkeypatch, dtype, full):
    from paper_2607_05583_gb300 import build
    build.build()
    rlm.load_library()
    B, L, D, M, K = 2, 333, 64, 16, 3
    inp = make_inputs(B, L, D, M, dtype, seed=5, with_dy=True)
    mx = make_mixer_inputs(inp, K, seed=6)
    p, x, dy, g = rlm.Params.from_arrays(*inp.params()), to_dev(inp.x, dtype), to_dev(inp.dy, dtype), to_dev(mx.g, dtype)
    s0 = torch.from_numpy(np.random.default_rng(7).standard_normal((3, B, D, M, 2)).astype(np.float32)).cuda()
    c_raw = np.random.default_rng(8).standard_normal((4, 4))

    def calls():
        empty = lambda: torch.zeros_like(x)
        state = lambda i: rlm.State(s0[i].clone(), torch.zeros(D, M, 4, device="cuda"))
        opt = lambda v: v if full else None
        ws = torch.empty(rlm.rlm_backward_workspace_size(B, L, D, M, x.dtype) + (64 << 20), dtype=torch.uint8, device="cuda")
        local, c = opt(rlm.Local.from_arrays(mx.conv_w, mx.scale)), opt(rlm.Coupling.from_arrays(c_raw, 0.5))
        conv = lambda: opt(rlm.ConvState(to_dev(mx.conv_in, dtype)))
        st, so, y = state(0), state(1), empty()
        rlm.rlm_mix_prefill(x, p, y, opt(so), workspace=opt(ws))
        y2 = empty()
        rlm.rlm_mix_prefill_from(x, p, opt(st), y2, opt(so), workspace=opt(ws))
        dx, gr, ds = empty(), rlm.Grads.empty(D, M), state(2)
        rlm.rlm_mix_backward(dy, x, p, dx, gr, workspace=opt(ws))
        dx2, gr2 = empty(), rlm.Grads.empty(D, M)
        rlm.rlm_mix_backward_from(dy, x, p, opt(state(0)), opt(state(1)), dx2, gr2, opt(ds), workspace=opt(ws))
        z, ci, co, sm = empty(), conv(), conv(), state(1)
        rlm.rlm_mixer_prefill(x, opt(g), p, local, z, conv_in=ci, state_out=opt(sm), conv_out=co, workspace=opt(ws),
                              state_in=opt(st), coupling=c)
        sd, cd = state(0), conv()
        rlm.rlm_state_init(sd, p)
        xt, gt, zt, yt = x[:, 0].contiguous(), g[:, 0].contiguous(), empty()[:, 0].contiguous(), empty()[:, 0].contiguous()
        rlm.rlm_mixer_decode(xt, opt(gt), sd, local, cd, zt, coupling=c)
        rlm.rlm_mix_decode(xt, sd, yt)
        torch.cuda.synchronize()
        out = [y, y2, dx, dx2, z, zt, yt, so.s, so.coef, ds.s, sm.s, sm.coef, sd.s]
        out += [getattr(q, k) for q in (gr, gr2) for k in ("decay", "freq", "amp", "phase")]
        return out + ([co.u, cd.u] if full else [])

    seen = []
    native = rlm._native

    class Watch:
        def __getattr__(self, name):
            f = getattr(native, name)

            def call(*args):
                status = f(*args)
                seen.append((name, status))
                return status
            return call

    monkeypatch.setattr(rlm, "_native", Watch())
    a = calls()
    assert {n for n, s in seen} == {"mix_prefill", "mix_backward", "mixer_prefill", "mixer_decode", "mix_decode"}
    assert all(s == 0 for _, s in seen)
    monkeypatch.setattr(rlm, "_native", rlm._CtypesOnly())
    b = calls()
    assert all(torch.equal(u, v) for u, v in zip(a, b))
