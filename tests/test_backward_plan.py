"""How the tcgen05 backward shares batch rows among its blocks: up to three levels of rows a
block.  The plan itself is checked on the CPU, the kernels on shapes picked by their plan."""
import ctypes

import numpy as np
import pytest

from synth import make_inputs
from tests._util import to_dev

torch = pytest.importorskip("torch")
rlm = pytest.importorskip("paper_2607_05583_gb300")

MAX_WALK = 16   # tiles


@pytest.fixture(scope="module")
def lib():
    from paper_2607_05583_gb300 import build
    build.build()
    return rlm.load_library()


def plan(lib, B, D, ntiles):
    """[(channel, first row, rows, level)] of every block."""
    out = (ctypes.c_int * 4)()
    n = lib.rlm_test_backward_plan(B, D, ntiles, -1, out)
    blocks = []
    for k in range(n):
        lib.rlm_test_backward_plan(B, D, ntiles, k, out)
        blocks.append(tuple(out))
    return blocks


def levels(blocks):
    """The plan's different numbers of rows a block, in the blocks' order of levels."""
    per = {}
    for _, _, n, lv in blocks:
        per[lv] = max(per.get(lv, 0), n)
    return [per[k] for k in sorted(per)]


def test_every_row_of_every_channel_is_taken_once(lib):
    rng = np.random.default_rng(0)
    seen = set()
    shapes = [(1, 8, 1), (2, 320, 1), (3, 320, 1), (16, 256, 4), (8, 256, 2), (64, 768, 1), (5, 1024, 3), (7, 64, 8), (4, 512, 16)]
    shapes += [(int(rng.integers(1, 41)), 8 * int(rng.integers(1, 80)), int(rng.integers(1, 10))) for _ in range(60)]
    for B, D, nt in shapes:
        blocks = plan(lib, B, D, nt)
        hits = np.zeros((D, B), int)
        for d, b0, n, _ in blocks:
            assert n == 1 or n * nt <= MAX_WALK
            hits[d, b0:b0 + n] += 1
            assert n >= 1 and b0 + n <= B
        assert (hits == 1).all(), (B, D, nt)
        lv = levels(blocks)
        assert lv == sorted(lv, reverse=True)
        seen.add(len(lv))
    assert {1, 2} <= seen


def shape_with(lib, want):
    """A small shape (B, D, 1 tile) whose plan has `want` levels on this device."""
    for B in range(2, 17):
        for D in range(64, 513, 8):
            lv = levels(plan(lib, B, D, 1))
            if len(lv) == want:
                return B, D, lv
    return None


def test_small_shapes_with_one_two_and_three_levels_exist(lib):
    for want in (1, 2, 3):
        assert shape_with(lib, want), want


def _states(B, D, M, seed):
    s = np.random.default_rng(seed).standard_normal((B, D, M, 2)).astype(np.float32)
    return rlm.State(torch.from_numpy(s).cuda(), torch.empty(D, M, 4, device="cuda"))


# Rows that share a block must give what they give alone: dx and d_state_in bit by bit, and
# gradients that are the rows' fp32 partials added with compensation.  Each of a
# gradient's B terms is rounded a few times (2^-24 each) on either side and the roundings
# are independent, so the two sums agree to 4 * 2^-24 in the l2 norm; sums kept in tensor
# memory over several rows (truncated additions) differ by several times that.
@pytest.mark.gpu
@pytest.mark.parametrize("case", ["two levels", "three levels", (8, 256, 4000, 16), (8, 256, 4096, 16), (40, 64, 100, 8),
                                  (6, 64, 4097, 32)])
def test_rows_in_blocks_of_several_levels(lib, case):
    if isinstance(case, str):
        B, D, _ = shape_with(lib, 2 if case.startswith("two") else 3)
        L, M = 131, 12
    else:
        B, D, L, M = case
    inp = make_inputs(B, L, D, M, "bf16", seed=B + L, with_dy=True)
    p = rlm.Params.from_arrays(*inp.params())
    x, dy = to_dev(inp.x, "bf16"), to_dev(inp.dy, "bf16")
    st, gs = _states(B, D, M, L), _states(B, D, M, L + 1)
    dx, gr, ds = torch.empty_like(x), rlm.Grads.empty(D, M), rlm.State.empty(B, D, M)
    rlm.rlm_mix_backward_from(dy, x, p, st, gs, dx, gr, ds)
    keys = ("decay", "freq", "amp", "phase")
    total = {k: torch.zeros(D, M, dtype=torch.float64, device="cuda") for k in keys}
    for b in range(B):
        one = lambda s: rlm.State(s.s[b:b + 1].contiguous(), s.coef)
        dx1, g1, ds1 = torch.empty_like(x[b:b + 1]), rlm.Grads.empty(D, M), rlm.State.empty(1, D, M)
        rlm.rlm_mix_backward_from(dy[b:b + 1].contiguous(), x[b:b + 1].contiguous(), p, one(st), one(gs), dx1, g1, ds1)
        assert torch.equal(dx1[0], dx[b]) and torch.equal(ds1.s[0], ds.s[b])
        for k in keys:
            total[k] += getattr(g1, k).double()
    for k in keys:
        err = (getattr(gr, k).double() - total[k]).norm() / total[k].norm()
        assert err <= 4 * 2.0 ** -24, (k, float(err))
