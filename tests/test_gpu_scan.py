"""Kernels at the edges of their tiles and splits.  The CUDA-core scan (fp32 with M > 16,
M > 32, a ragged length from a state, fp32 backward): chunks of 64 tokens, tiles of 1024,
mode groups of 8, 16, 32 and 64, segments of whole tiles, batch rows that share a tile.
The tcgen05 backward with several rows per block, and the coupled decode step with
several blocks per row.  Tolerances are the operator's parity bar unless said."""
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


def _state(B, D, M, seed):
    rng = np.random.default_rng(seed)
    s = (3.0 * rng.standard_normal((B, D, M, 2))).astype(np.float32)
    st = rlm.State(torch.from_numpy(s).cuda(), torch.empty(D, M, 4, device="cuda"))
    return st, s[..., 0].astype(np.float64) + 1j * s[..., 1]


# Lengths at chunk and tile edges; the last two rows are long enough for several segments
# (B * D / 4 blocks against a few hundred resident ones).
@pytest.mark.parametrize("B,L,D,M,dtype", [
    (2, 1, 16, 9, "f32"), (1, 63, 8, 33, "f32"), (3, 65, 16, 17, "f32"), (2, 127, 8, 64, "bf16"),
    (2, 1023, 16, 8, "bf16"), (1, 1025, 24, 1, "f32"), (2, 1087, 8, 16, "bf16"), (1, 2049, 16, 32, "f32"),
    (1, 20001, 8, 5, "f32"), (1, 9999, 8, 40, "bf16"),
    # several batch rows in a tile (at most 4 or 8 chunks), the last tile partly empty
    (5, 100, 8, 16, "bf16"), (6, 255, 16, 3, "f32"), (3, 257, 8, 20, "f32"), (5, 511, 8, 33, "f32"),
])
def test_prefill_from_a_state_at_tile_edges(B, L, D, M, dtype):
    inp = make_inputs(B, L, D, M, dtype, seed=L + M)
    x = to_dev(inp.x, dtype)
    p = rlm.Params.from_arrays(*inp.params())
    st, s0 = _state(B, D, M, L)
    y = torch.full_like(x, float("nan"))
    # In place: the terminal state overwrites the initial one.
    rlm.rlm_mix_prefill_from(x, p, st, y, st)
    torch.cuda.synchronize()
    y_ref, s_ref = oracle.rec_prefill(inp.x, *inp.params(), state_in=s0)
    assert_close(to_np(y), y_ref, TOL[dtype], "y")
    s = st.complex().cpu().numpy()
    assert_close(s.real, s_ref.real, TOL["f32"], "state re")
    assert_close(s.imag, s_ref.imag, TOL["f32"], "state im")


# The terminal state of a sequence that ends inside a chunk: its powers are shared out among
# four lanes and two halves of the table (n < 32 and above), with one, two or four batch
# rows in a tile and the end in a first, middle or second tile.
@pytest.mark.parametrize("tail", [2, 31, 32, 33, 62])
@pytest.mark.parametrize("B,chunks,M", [(5, 0, 16), (3, 6, 8), (1, 9, 32), (2, 17, 64)])
def test_terminal_state_of_a_partial_chunk(B, chunks, M, tail):
    L, D = 64 * chunks + tail, 8
    inp = make_inputs(B, L, D, M, "f32", seed=L + M)
    st, s0 = _state(B, D, M, L)
    x = to_dev(inp.x, "f32")
    y, so = torch.empty_like(x), rlm.State.empty(B, D, M)
    rlm.rlm_mix_prefill_from(x, rlm.Params.from_arrays(*inp.params()), st, y, so)
    torch.cuda.synchronize()
    y_ref, s_ref = oracle.rec_prefill(inp.x, *inp.params(), state_in=s0)
    assert_close(to_np(y), y_ref, TOL["f32"], "y")
    s = so.complex().cpu().numpy()
    assert_close(s.real, s_ref.real, TOL["f32"], "state re")
    assert_close(s.imag, s_ref.imag, TOL["f32"], "state im")


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
@pytest.mark.parametrize("t", [0, 70, 1030])
def test_a_non_finite_drive_leaves_earlier_outputs_alone(bad, t):
    B, L, D, M = 1, 1200, 8, 20
    inp = make_inputs(B, L, D, M, "f32", seed=3)
    p = rlm.Params.from_arrays(*inp.params())
    x = to_dev(inp.x, "f32")
    y0, y1 = torch.empty_like(x), torch.empty_like(x)
    rlm.rlm_mix_prefill(x, p, y0)
    x[0, t, 2] = bad
    rlm.rlm_mix_prefill(x, p, y1)
    other = [c for c in range(D) if c != 2]
    assert torch.equal(y0[..., other], y1[..., other])
    # The guarded and the plain product add in the same order up to rounding.
    assert_close(to_np(y1[0, :t, 2]), to_np(y0[0, :t, 2]), 1e-5) if t else None
    assert not torch.isfinite(y1[0, t, 2])


@pytest.mark.parametrize("B,L,D,M,dtype", [
    (1, 1, 8, 4, "f32"), (2, 63, 8, 8, "f32"), (1, 64, 16, 16, "f32"), (2, 100, 8, 33, "bf16"),
    (2, 1024, 8, 17, "f32"), (1, 1090, 16, 32, "f32"), (1, 12345, 8, 9, "f32"), (1, 4096, 8, 64, "f32"),
    (9, 74, 8, 16, "f32"), (4, 256, 16, 32, "f32"), (3, 300, 8, 5, "f32"), (5, 512, 8, 40, "bf16"),
])
def test_backward_with_state_terms_at_tile_edges(B, L, D, M, dtype):
    inp = make_inputs(B, L, D, M, dtype, seed=L + 3 * M, with_dy=True)
    p = rlm.Params.from_arrays(*inp.params())
    x, dy = to_dev(inp.x, dtype), to_dev(inp.dy, dtype)
    (st, s0), (gs, g) = _state(B, D, M, L), _state(B, D, M, L + 1)
    dx, gr, ds = torch.empty_like(x), rlm.Grads.empty(D, M), rlm.State.empty(B, D, M)
    rlm.rlm_mix_backward_from(dy, x, p, st, gs, dx, gr, ds)
    torch.cuda.synchronize()
    ref = oracle.backward_rec(inp.x, inp.dy, *inp.params(), state_in=s0, d_state_out=g)
    assert_close(to_np(dx), ref[0], TOL[dtype], "dx")
    for k in ("decay", "freq", "amp", "phase"):
        assert_close(getattr(gr, k).cpu().numpy(), ref[1][k], TOL["f32"], k)
    d = ds.complex().cpu().numpy()
    assert_close(d.real, ref[1]["state_in"].real, TOL["f32"], "d_state re")
    assert_close(d.imag, ref[1]["state_in"].imag, TOL["f32"], "d_state im")


# The tensor-core backward with several rows of a channel per block: one level of rows
# (many short rows), three levels (few tiles, more blocks than fit at once), a ragged
# length, and one row per block.  Rows must not see one another's carry: dx of each row
# equals the row's own backward, and the gradients are the rows' sum.
@pytest.mark.parametrize("B,L,D,M", [(7, 130, 96, 32), (40, 100, 64, 16), (9, 2049, 256, 8), (3, 64, 8, 1)])
def test_backward_rows_sharing_a_block(B, L, D, M):
    inp = make_inputs(B, L, D, M, "bf16", seed=B + L, with_dy=True)
    p = rlm.Params.from_arrays(*inp.params())
    x, dy = to_dev(inp.x, "bf16"), to_dev(inp.dy, "bf16")
    (st, _), (gs, _) = _state(B, D, M, L), _state(B, D, M, L + 1)
    dx, gr, ds = torch.empty_like(x), rlm.Grads.empty(D, M), rlm.State.empty(B, D, M)
    rlm.rlm_mix_backward_from(dy, x, p, st, gs, dx, gr, ds)
    total = {k: torch.zeros(D, M, dtype=torch.float64, device="cuda") for k in ("decay", "freq", "amp", "phase")}
    for b in range(B):
        one = lambda s: rlm.State(s.s[b:b + 1].contiguous(), s.coef)
        dx1, g1, ds1 = torch.empty_like(x[b:b + 1]), rlm.Grads.empty(D, M), rlm.State.empty(1, D, M)
        rlm.rlm_mix_backward_from(dy[b:b + 1].contiguous(), x[b:b + 1].contiguous(), p, one(st), one(gs), dx1, g1, ds1)
        assert torch.equal(dx1[0], dx[b]) and torch.equal(ds1.s[0], ds.s[b])
        for k in total:
            total[k] += getattr(g1, k).double()
    for k in total:
        # fp32 sums of the same terms in another order.
        assert_close(getattr(gr, k).cpu().numpy(), total[k].cpu().numpy(), 2e-5, k)


# The coupled decode step split over blocks of a row: 8, 4, 2 and 1 blocks (few or many
# rows, narrow heads, few modes), one head, odd head widths per block, K from 0 to 8.
@pytest.mark.parametrize("B,D,M,H,K,dtype", [
    (1, 256, 16, 8, 4, "bf16"), (3, 512, 8, 16, 8, "f32"), (70, 256, 16, 8, 2, "bf16"), (90, 256, 16, 8, 4, "bf16"),
    (2, 64, 64, 1, 1, "f32"), (5, 120, 32, 5, 3, "f32"), (4, 48, 32, 4, 4, "bf16"), (2, 8, 2, 8, 4, "f32"),
])
def test_coupled_decode_split_over_blocks(B, D, M, H, K, dtype):
    inp = make_inputs(B, 4, D, M, dtype, seed=B + D + K)
    mx = make_mixer_inputs(inp, K, seed=B + M)
    c_raw = np.random.default_rng(H).standard_normal((H, H))
    x, g = to_dev(inp.x, dtype), to_dev(mx.g, dtype)
    p = rlm.Params.from_arrays(*inp.params())
    local = rlm.Local.from_arrays(mx.conv_w, mx.scale) if K else None
    st = rlm.State.empty(B, D, M)
    rlm.rlm_state_init(st, p)
    cs = rlm.ConvState(to_dev(mx.conv_in, dtype)) if K > 1 else None
    zs = []
    for t in range(4):
        z = torch.full_like(x[:, t], float("nan"))
        rlm.rlm_mixer_decode(x[:, t].contiguous(), g[:, t].contiguous(), st, local, cs, z,
                             coupling=rlm.Coupling.from_arrays(c_raw, 0.5))
        zs.append(z)
    torch.cuda.synchronize()
    zr, sr, tr = oracle.mixer_prefill(inp.x, mx.g, *inp.params(), mx.conv_w, mx.scale,
                                      conv_in=mx.conv_in if K > 1 else None, coupling=(c_raw, 0.5))
    assert_close(to_np(torch.stack(zs, 1)), zr, TOL[dtype], "z")
    s = st.complex().cpu().numpy()
    assert_close(s.real, sr.real, TOL["f32"], "state re")
    assert_close(s.imag, sr.imag, TOL["f32"], "state im")
    if K > 1:
        np.testing.assert_array_equal(to_np(cs.u), tr)
