"""Short sequences on the CUDA cores: the recurrence up to 8 tokens, and the scan's narrow
tiles (4 chunks of 64 tokens, several batch rows in a tile up to 2 chunks, two warps a
channel above 32 modes) at their edges: a partial chunk alone, whole chunks, several tiles, the
mode groups of 8, 16, 32 and 64.  Against the fp64 oracle at the operator's parity bar, and
at a bar of 2e-6 for fp32: sums of at most a few hundred roundings of 6e-8 that mostly cancel."""
import numpy as np
import pytest

import oracle
from synth import make_inputs
from tests._util import TOL, assert_close, to_dev, to_np

torch = pytest.importorskip("torch")
rlm = pytest.importorskip("paper_2607_05583_gb300")

pytestmark = pytest.mark.gpu

FINE = {"f32": 2e-6, "bf16": TOL["bf16"]}
SHAPES = [(B, L, D, M, dtype) for L, rows in [
    (1, 3), (2, 1), (5, 2), (7, 70), (8, 5), (9, 3), (15, 4), (16, 1), (17, 5), (31, 2), (32, 3), (33, 9), (48, 1),
    (49, 4), (63, 6), (64, 5), (65, 3), (127, 2), (128, 5), (129, 1), (191, 2), (192, 3), (256, 1), (257, 2), (300, 1),
    (511, 1), (513, 1)]
    for B, D, M, dtype in [(rows, 8, (1, 8, 9, 16, 17, 31, 32, 33, 47, 64)[(L + rows) % 10], "f32"),
                           (rows, 16, (64, 33, 5, 24, 16, 1, 40, 32)[(L + rows) % 8], ("f32", "bf16")[L % 2])]]


@pytest.fixture(scope="module", autouse=True)
def lib():
    from paper_2607_05583_gb300 import build
    build.build()
    return rlm.load_library()


def _state(B, D, M, seed):
    s = np.random.default_rng(seed).standard_normal((B, D, M, 2)).astype(np.float32)
    return rlm.State(torch.from_numpy(s).cuda(), torch.empty(D, M, 4, device="cuda")), s[..., 0].astype(np.float64) + 1j * s[..., 1]


def _complex(got, ref, what):
    g = got.complex().cpu().numpy()
    assert_close(g.real, ref.real, FINE["f32"], what + " re")
    assert_close(g.imag, ref.imag, FINE["f32"], what + " im")


# (fp32 prefills of up to 16 modes and whole chunks run on the tensor cores, which have a bar of their own.)
@pytest.mark.parametrize("B,L,D,M,dtype", [s for s in SHAPES if s[1] % 64 or s[3] > 16 or s[4] == "bf16"])
def test_short_prefill_from_a_state(B, L, D, M, dtype):
    inp = make_inputs(B, L, D, M, dtype, seed=7 * L + M)
    p, x = rlm.Params.from_arrays(*inp.params()), to_dev(inp.x, dtype)
    st, s0 = _state(B, D, M, L)
    y = torch.full_like(x, float("nan"))
    rlm.rlm_mix_prefill_from(x, p, st, y, st)   # in place
    torch.cuda.synchronize()
    y_ref, s_ref = oracle.rec_prefill(inp.x, *inp.params(), state_in=s0)
    assert_close(to_np(y), y_ref, FINE[dtype], "y")
    _complex(st, s_ref, "state")


@pytest.mark.parametrize("states", [True, False])
@pytest.mark.parametrize("B,L,D,M,dtype", [s for s in SHAPES if s[4] == "f32" or s[3] > 32])
def test_short_backward(B, L, D, M, dtype, states):
    inp = make_inputs(B, L, D, M, dtype, seed=5 * L + M, with_dy=True)
    p, x, dy = rlm.Params.from_arrays(*inp.params()), to_dev(inp.x, dtype), to_dev(inp.dy, dtype)
    dx, gr, ds = torch.full_like(x, float("nan")), rlm.Grads.empty(D, M), rlm.State.empty(B, D, M)
    if states:
        (st, s0), (gs, g) = _state(B, D, M, L), _state(B, D, M, L + 1)
        rlm.rlm_mix_backward_from(dy, x, p, st, gs, dx, gr, ds)
        ref = oracle.backward_rec(inp.x, inp.dy, *inp.params(), state_in=s0, d_state_out=g)
        _complex(ds, ref[1]["state_in"], "d_state")
    else:
        rlm.rlm_mix_backward(dy, x, p, dx, gr)
        ref = oracle.backward_rec(inp.x, inp.dy, *inp.params())
    assert_close(to_np(dx), ref[0], FINE[dtype], "dx")
    for k in ("decay", "freq", "amp", "phase"):
        if np.abs(ref[1][k]).max() > 0:   # (one token: dgamma and domega may vanish)
            assert_close(getattr(gr, k).cpu().numpy(), ref[1][k], 5 * FINE["f32"], k)
        else:
            assert not getattr(gr, k).any()


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
@pytest.mark.parametrize("L,t", [(5, 2), (40, 20), (200, 70), (200, 130), (400, 300)])
@pytest.mark.parametrize("M", [4, 20, 40])
def test_a_non_finite_drive_leaves_earlier_tokens_and_other_rows_alone(bad, L, t, M):
    B, D = 3, 8
    inp = make_inputs(B, L, D, M, "f32", seed=L + M, with_dy=True)
    p, x = rlm.Params.from_arrays(*inp.params()), to_dev(inp.x, "f32")
    y0, y1 = torch.empty_like(x), torch.empty_like(x)
    s0, s1 = rlm.State.empty(B, D, M), rlm.State.empty(B, D, M)
    zero = rlm.State(torch.zeros(B, D, M, 2, device="cuda"), torch.empty(D, M, 4, device="cuda"))
    rlm.rlm_mix_prefill_from(x, p, zero, y0, s0)
    x[1, t, 2] = bad
    rlm.rlm_mix_prefill_from(x, p, zero, y1, s1)
    others = [(b, c) for b in range(B) for c in range(D) if (b, c) != (1, 2)]
    for b, c in others:
        assert torch.equal(y0[b, :, c], y1[b, :, c]) and torch.equal(s0.s[b, c], s1.s[b, c])
    assert torch.isfinite(y1[1, :t, 2]).all() and not torch.isfinite(y1[1, t, 2])
    assert_close(to_np(y1[1, :t, 2]), to_np(y0[1, :t, 2]), 1e-5)
    # Reverse time: dx after a bad dy stays clean.
    dy = to_dev(inp.dy, "f32")
    x = to_dev(inp.x, "f32")
    d0, d1, gr = torch.empty_like(x), torch.empty_like(x), rlm.Grads.empty(D, M)
    rlm.rlm_mix_backward(dy, x, p, d0, gr)
    dy[1, t, 2] = bad
    rlm.rlm_mix_backward(dy, x, p, d1, gr)
    for b, c in others:
        assert torch.equal(d0[b, :, c], d1[b, :, c])
    assert torch.isfinite(d1[1, t + 1:, 2]).all() and not torch.isfinite(d1[1, t, 2])
    assert_close(to_np(d1[1, t + 1:, 2]), to_np(d0[1, t + 1:, 2]), 1e-5)
