"""Workloads of the resonant mixing library for timing and comparison.

Each case is one pass through the public entry points as a program would make it: a
decode step, a captured run of mixer decode steps, prompts of several lengths, a
continued prompt, the mixer over a sequence, and training steps (forward, backward).
The sizes are those of the repository's configurations (the 6M layer, the long-context
prefill, the D = 512 / M = 32 training layer, the small fp32 problem) or lie between
them; parameters follow the same distributions (decay U[0.001, 0.1], frequency
U[0, pi], amplitude N(0, 1/M), phase U[0, 2 pi), drives N(0, 1)).
"""
import math

import torch

import paper_2607_05583_gb300 as rlm

_DTYPE = {"bf16": torch.bfloat16, "f32": torch.float32}


def listed():
    return [
        # One token of an interactive session, called eagerly: the smallest call.
        dict(name="decode_step", kind="decode", B=1, D=256, M=16, dtype="bf16", steps=1, graph=False, mixer=False,
             gate=False, K=0, H=0),
        # A serving loop: a captured run of steps of the whole mixer at batch 64.
        dict(name="mixer_decode_graph", kind="decode", B=64, D=256, M=16, dtype="bf16", steps=32, graph=True,
             mixer=True, gate=True, K=4, H=8),
        # The small fp32 problem: a short single sequence.
        dict(name="prompt_small_f32", kind="prefill", B=1, L=256, D=64, M=4, dtype="f32", state_in=False,
             state_out=True),
        # The 6M model's layer over a batch of prompts.
        dict(name="prompt_6m_layer", kind="prefill", B=8, L=2048, D=256, M=16, dtype="bf16", state_in=False,
             state_out=True),
        # Long-context prefill.
        dict(name="prompt_long", kind="prefill", B=4, L=32768, D=256, M=16, dtype="bf16", state_in=False,
             state_out=True),
        # A single odd-length prompt through the wider, 32-mode layer.
        dict(name="prompt_single_m32", kind="prefill", B=1, L=12289, D=512, M=32, dtype="bf16", state_in=False,
             state_out=True),
        # The next turn of a conversation: a prompt that continues from kept states.
        dict(name="prompt_continued", kind="prefill", B=8, L=1000, D=256, M=16, dtype="bf16", state_in=True,
             state_out=True),
        # A full-precision forward over long sequences.
        dict(name="prompt_f32", kind="prefill", B=4, L=8192, D=256, M=16, dtype="f32", state_in=False,
             state_out=True),
        # The whole mixer (gate, local path, head coupling) over long prompts.
        dict(name="mixer_prompt", kind="mixer", B=4, L=8192, D=256, M=16, dtype="bf16", gate=True, K=4, H=8,
             history=True),
        # One training step of the wide layer: forward, then dx and the parameter gradients.
        dict(name="train_step", kind="train", B=4, L=32768, D=512, M=32, dtype="bf16"),
        # The same layer trained (or its gradients checked) in full precision.
        dict(name="train_step_f32", kind="train", B=2, L=4096, D=512, M=32, dtype="f32"),
        # Truncated back-propagation through time: a segment that starts from a state and
        # whose terminal state has a gradient.
        dict(name="backward_states", kind="backward_from", B=8, L=4096, D=256, M=16, dtype="bf16"),
    ]


def _between(rng, lo, hi):
    """An integer spread over the logarithm of lo..hi."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["decode", "prefill", "prefill", "prefill", "mixer", "train", "train", "backward_from"])
    dtype = rng.choice(["bf16", "bf16", "f32"])
    D = 8 * _between(rng, 8, 96)
    M = rng.choice([1, 2, 4, 8, 16, 16, 32, 32, _between(rng, 1, 64)])
    if kind == "decode":
        mixer = rng.random() < 0.5
        return dict(kind=kind, B=_between(rng, 1, 256), D=D, M=M, dtype=dtype, steps=_between(rng, 1, 32),
                    graph=rng.random() < 0.5, mixer=mixer, gate=mixer, K=rng.randint(0, 4) if mixer else 0,
                    H=rng.choice([0, 4, 8]) if mixer else 0)
    # Token-channels between the small problem's and the largest listed case's (fp32
    # and many modes cost more a piece, so they stop earlier).
    most = 4 * 32768 * 512
    if dtype == "f32" or M > 32:
        most //= 16
    elif kind == "backward_from":
        most //= 2
    L = _between(rng, 64, 32768)
    L = min(L, max(64, most // D))
    B = _between(rng, 1, max(1, min(64, most // (L * D))))
    case = dict(kind=kind, B=B, L=L, D=D, M=M, dtype=dtype)
    if kind == "prefill":
        case.update(state_in=rng.random() < 0.4, state_out=True)
    elif kind == "mixer":
        case.update(gate=True, K=rng.randint(0, 4), H=rng.choice([0, 4, 8]), history=rng.random() < 0.5)
    return case


# ------------------------------------------------------------------ inputs
def _inputs(case, seed):
    """The tensors of a case, from its seed alone."""
    B, D, M = case["B"], case["D"], case["M"]
    dt = _DTYPE[case["dtype"]]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)

    def normal(*shape, dtype=torch.float32, scale=1.0):
        return (torch.randn(*shape, generator=gen, device="cuda", dtype=torch.float32) * scale).to(dtype)

    def uniform(lo, hi, *shape):
        return torch.rand(*shape, generator=gen, device="cuda", dtype=torch.float32) * (hi - lo) + lo

    t = {"decay": uniform(0.001, 0.1, D, M), "freq": uniform(0.0, math.pi, D, M),
         "amp": normal(D, M, scale=M ** -0.5), "phase": uniform(0.0, 2 * math.pi, D, M)}
    kind = case["kind"]
    tokens = case["steps"] if kind == "decode" else case["L"]
    # Decode takes one [B][1][D] field a step; its tokens are kept step by step.
    t["x"] = normal(tokens, B, 1, D, dtype=dt) if kind == "decode" else normal(B, tokens, D, dtype=dt)
    if kind in ("train", "backward_from"):
        t["dy"] = normal(B, tokens, D, dtype=dt)
    if kind == "decode" or case.get("state_in") or kind == "backward_from":
        # A state that a prompt leaves: its variance is about 1 / (2 gamma) a mode.
        t["s"] = normal(B, D, M, 2, scale=3.0)
    if kind == "backward_from":
        t["g"] = normal(B, D, M, 2)
    if case.get("gate"):
        t["gate"] = normal(*t["x"].shape, dtype=dt)
    K, H = case.get("K", 0), case.get("H", 0)
    if K:
        t["conv_w"], t["scale"] = normal(D, K, scale=K ** -0.5), uniform(0.5, 1.5, D)
        if K > 1 and (kind == "decode" or case.get("history")):
            t["conv"] = normal(B, K - 1, D, dtype=dt)
    if H:
        t["c_raw"] = normal(H, H)
    return t


_COUPLING = 0.5


def prepare(case, seed):
    B, D, M = case["B"], case["D"], case["M"]
    dt = _DTYPE[case["dtype"]]
    t = _inputs(case, seed)
    st = {"case": case, "params": rlm.Params(t["decay"], t["freq"], t["amp"], t["phase"]), "x": t["x"],
          "gate": t.get("gate")}
    st["local"] = rlm.Local(t["conv_w"], t["scale"]) if "conv_w" in t else None
    st["coupling"] = rlm.Coupling(t["c_raw"], _COUPLING) if "c_raw" in t else None
    st["conv"] = rlm.ConvState(t["conv"]) if "conv" in t else None
    if case["kind"] == "decode":
        st["state"] = rlm.State.empty(B, D, M)
        rlm.rlm_state_init(st["state"], st["params"])
        st["state"].s.copy_(t["s"])
        st["y"] = torch.empty_like(t["x"])
        # Fields of one token are sliced once, as a program with fixed buffers has them.
        st["tokens"] = [(st["x"][i], st["gate"][i] if st["gate"] is not None else None, st["y"][i])
                        for i in range(case["steps"])]
        if case["graph"]:
            # Capturing records the steps without running them.
            st["graph"] = torch.cuda.CUDAGraph()
            side = torch.cuda.Stream()
            side.wait_stream(torch.cuda.current_stream())
            torch.cuda.synchronize()
            with torch.cuda.stream(side):
                st["graph"].capture_begin()
                _decode(st)
                st["graph"].capture_end()
            torch.cuda.current_stream().wait_stream(side)
        return st
    L = case["L"]
    st["y"] = torch.empty_like(t["x"])
    st["state_in"] = rlm.State(t["s"], torch.empty(D, M, 4, device="cuda")) if "s" in t else None
    if case["kind"] in ("train", "backward_from"):
        st["dy"], st["dx"] = t["dy"], torch.empty_like(t["x"])
        st["grads"] = rlm.Grads.empty(D, M)
        need = max(rlm.rlm_prefill_workspace_size(B, L, D, M, dt), rlm.rlm_backward_workspace_size(B, L, D, M, dt))
        st["workspace"] = torch.empty(max(need, 256), dtype=torch.uint8, device="cuda")
        if case["kind"] == "backward_from":
            st["g"] = rlm.State(t["g"], torch.empty(D, M, 4, device="cuda"))
            st["d_state"] = rlm.State.empty(B, D, M)
    else:
        st["state_out"] = rlm.State.empty(B, D, M)
        if case["kind"] == "mixer" and case["K"] > 1:
            st["conv_out"] = rlm.ConvState.empty(B, D, case["K"], dtype=dt)
    return st


def _decode(st):
    if st["case"]["mixer"]:
        for x, g, y in st["tokens"]:
            rlm.rlm_mixer_decode(x, g, st["state"], st["local"], st["conv"], y, coupling=st["coupling"])
    else:
        for x, _, y in st["tokens"]:
            rlm.rlm_mix_decode(x, st["state"], y)


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "decode":
        if "graph" in st:
            st["graph"].replay()
        else:
            _decode(st)
        return {"y": st["y"], "s": st["state"].s, "conv": st["conv"].u if st["conv"] is not None else None}
    if kind == "prefill":
        so = st["state_out"]
        if st["state_in"] is not None:
            rlm.rlm_mix_prefill_from(st["x"], st["params"], st["state_in"], st["y"], so)
        else:
            rlm.rlm_mix_prefill(st["x"], st["params"], st["y"], so)
        return {"y": st["y"], "s": so.s, "coef": so.coef}
    if kind == "mixer":
        so, co = st["state_out"], st.get("conv_out")
        rlm.rlm_mixer_prefill(st["x"], st["gate"], st["params"], st["local"], st["y"], conv_in=st["conv"],
                              state_out=so, conv_out=co, coupling=st["coupling"])
        return {"y": st["y"], "s": so.s, "coef": so.coef, "conv": co.u if co is not None else None}
    gr = st["grads"]
    out = {"dx": st["dx"], "decay": gr.decay, "freq": gr.freq, "amp": gr.amp, "phase": gr.phase}
    if kind == "train":
        rlm.rlm_mix_prefill(st["x"], st["params"], st["y"], workspace=st["workspace"])
        rlm.rlm_mix_backward(st["dy"], st["x"], st["params"], st["dx"], gr, workspace=st["workspace"])
        out["y"] = st["y"]
    else:
        rlm.rlm_mix_backward_from(st["dy"], st["x"], st["params"], st["state_in"], st["g"], st["dx"], gr,
                                  st["d_state"], workspace=st["workspace"])
        out["d_state"] = st["d_state"].s
    return out


# -------------------------------------------------------------------- work
def work(case):
    """Bytes: every input read once and every output written once.  Flops: the chunk-free
    recurrence (a complex multiply-add and a readout, 10 a mode and token-channel; the
    backward carries two such recurrences and forms two products)."""
    B, D, M = case["B"], case["D"], case["M"]
    e = 2 if case["dtype"] == "bf16" else 4
    kind = case["kind"]
    n = B * D * (case["steps"] if kind == "decode" else case["L"])
    state, modes = 8 * B * D * M, 16 * D * M
    K, H = case.get("K", 0), case.get("H", 0)
    fields = 2 + (1 if case.get("gate") else 0)
    flops = 10 * n * M + (2 * K + 2 * H) * n
    if kind == "decode":
        history = 2 * B * D * max(K - 1, 0) * e
        return {"bytes": n * fields * e + case["steps"] * (2 * state + modes + history), "flops": flops}
    if kind in ("prefill", "mixer"):
        states = state * (2 if case.get("state_in") else 1)
        return {"bytes": n * fields * e + states + 2 * modes, "flops": flops}
    if kind == "train":
        return {"bytes": n * 5 * e + 3 * modes, "flops": flops + 26 * n * M}
    return {"bytes": n * 3 * e + 3 * state + 2 * modes, "flops": 26 * n * M}


# ------------------------------------------------------- the same in 64 bits
def _powers(lam, n0, n):
    """lambda^(n0 + i), i < n, as [D][n][M]."""
    i = torch.arange(n0, n0 + n, device=lam.device, dtype=torch.float64)
    return torch.exp(torch.log(lam)[:, None, :] * i[None, :, None])


def _toward_end(x, lam, jordan=False):
    """sum_j lambda^(L-1-j) x_j per (b, d, m) for x [B][L][D]; with jordan the sums
    weighted by L-1-j as well."""
    B, L, D = x.shape
    xt = x.permute(2, 0, 1)
    s = torch.zeros(D, B, lam.shape[1], dtype=torch.complex128, device=x.device)
    r = torch.zeros_like(s)
    step = 1024
    for j0 in range(0, L, step):
        j1 = min(L, j0 + step)
        p = _powers(lam, L - j1, j1 - j0).flip(1)
        seg = xt[:, :, j0:j1].contiguous()
        s += torch.complex(torch.bmm(seg, p.real.contiguous()), torch.bmm(seg, p.imag.contiguous()))
        if jordan:
            p = p * torch.arange(L - 1 - j0, L - 1 - j1, -1, device=x.device, dtype=torch.float64)[None, :, None]
            r += torch.complex(torch.bmm(seg, p.real.contiguous()), torch.bmm(seg, p.imag.contiguous()))
    return s.permute(1, 0, 2), r.permute(1, 0, 2)


def _response(weight, lam, n0, n):
    """Re(sum_m weight lambda^(n0 + i)) for weight [B][D][M]: [B][n][D]."""
    B, D, M = weight.shape
    w = weight.permute(1, 0, 2)
    out = torch.empty(D, B, n, dtype=torch.float64, device=lam.device)
    step = 1024
    for i0 in range(0, n, step):
        i1 = min(n, i0 + step)
        p = _powers(lam, n0 + i0, i1 - i0)
        pr, pi = p.real.transpose(1, 2).contiguous(), p.imag.transpose(1, 2).contiguous()
        out[:, :, i0:i1] = torch.bmm(w.real.contiguous(), pr) - torch.bmm(w.imag.contiguous(), pi)
    return out.permute(1, 2, 0)


def _channels(D, L, B):
    """Channels a piece whose transforms stay within a few GB."""
    return max(1, min(D, int(2e9 // (32 * B * max(L, 1)))))


def _conv(x, k, causal=True):
    """Causal (or anti-causal) convolution of x [B][L][D] with k [D][L]."""
    B, L, D = x.shape
    out = torch.empty_like(x)
    step = _channels(D, L, B)
    for d in range(0, D, step):
        f = torch.fft.rfft(x[:, :, d:d + step].permute(0, 2, 1), n=2 * L)
        h = torch.fft.rfft(k[d:d + step], n=2 * L)
        out[:, :, d:d + step] = torch.fft.irfft(f * (h if causal else h.conj()), n=2 * L)[..., :L].permute(0, 2, 1)
    return out


def _lags(x, dy):
    """rho[d][n] = sum_b sum_j x_j dy_{j+n}."""
    B, L, D = x.shape
    out = torch.empty(D, L, dtype=torch.float64, device=x.device)
    step = _channels(D, L, B)
    for d in range(0, D, step):
        f = torch.fft.rfft(x[:, :, d:d + step].permute(0, 2, 1), n=2 * L)
        h = torch.fft.rfft(dy[:, :, d:d + step].permute(0, 2, 1), n=2 * L)
        out[d:d + step] = torch.fft.irfft((f.conj() * h).sum(0), n=2 * L)[..., :L]
    return out


def _pair(z):
    return torch.view_as_real(z.resolve_conj().contiguous())


def exact(case, seed):
    t = _inputs(case, seed)
    kind = case["kind"]
    decay, freq, amp, phase = (t[k].double() for k in ("decay", "freq", "amp", "phase"))
    lam = torch.exp(torch.complex(-decay, freq))
    c = torch.polar(torch.ones_like(amp), phase) * amp
    coef = torch.stack([lam.real, lam.imag, c.real, c.imag], -1)
    K, H = case.get("K", 0), case.get("H", 0)
    x = t["x"].double()
    gate = torch.sigmoid(t["gate"].double()) if "gate" in t else None
    s_in = torch.view_as_complex(t["s"].double()) if "s" in t else None
    couple = None
    if H:
        couple = torch.eye(H, dtype=torch.float64, device="cuda") + _COUPLING / H ** 0.5 * torch.tanh(t["c_raw"].double())

    def mixed(y, u, g):
        """The mixer around y [B][L][D]; u holds K - 1 earlier drives, then the L drives."""
        B, L, D = y.shape
        if couple is not None:
            y = torch.einsum("gh,blhi->blgi", couple, y.reshape(B, L, H, D // H)).reshape(B, L, D)
        if g is not None:
            y = g * y
        if K:
            w, scale = t["conv_w"].double(), t["scale"].double()
            y = y + scale * sum(w[:, k] * u[:, K - 1 - k:K - 1 - k + L] for k in range(K))
        return y

    if kind == "decode":
        s, hist, ys = s_in, t["conv"].double() if "conv" in t else x.new_zeros(case["B"], 0, case["D"]), []
        for i in range(case["steps"]):
            s = lam * s + x[i].transpose(1, 2)
            y = (c * s).real.sum(-1)[:, None]
            if case["mixer"]:
                u = torch.cat([hist, x[i]], 1)
                y = mixed(y, u, gate[i] if gate is not None else None)
                hist = u[:, 1:] if K > 1 else hist
            ys.append(y)
        return {"y": torch.stack(ys), "s": _pair(s), "conv": hist if "conv" in t else None}

    B, L, D = x.shape
    kern = _response(c[None], lam, 0, L)[0].T.contiguous()
    if kind in ("prefill", "mixer"):
        y = _conv(x, kern)
        s = _toward_end(x, lam)[0]
        if s_in is not None:
            y = y + _response(c * lam * s_in, lam, 0, L)
            s = s + lam ** L * s_in
        out = {"y": y, "s": _pair(s), "coef": coef}
        if kind == "mixer":
            past = t["conv"].double() if "conv" in t else x.new_zeros(B, max(K - 1, 0), D)
            u = torch.cat([past, x], 1)
            out["y"] = mixed(y, u, gate)
            out["conv"] = u[:, L:] if K > 1 else None
        return out

    dy = t["dy"].double()
    dx = _conv(dy, kern, causal=False)
    rho = _lags(x, dy)
    # sum_n lambda^n rho[n] and sum_n n lambda^n rho[n]: rho reversed toward its end.
    G, P = (v[0] for v in _toward_end(rho.T.flip(0)[None].contiguous(), lam, jordan=True))
    out = {}
    if kind == "backward_from":
        g = torch.view_as_complex(t["g"].double())
        S0, R0 = _toward_end(dy.flip(1), lam, jordan=True)
        G = G + (s_in * lam * S0).sum(0)
        P = P + (s_in * lam * (R0 + S0)).sum(0)
        lamL = lam ** L
        J = _toward_end(x, lam, jordan=True)[1] + L * lamL * s_in
        J = (g.conj() * J).sum(0)
        dx = dx + _response(g.conj(), lam, 0, L).flip(1)
        out["d_state"] = _pair((c * lam * S0).conj() + g * lamL.conj())
    else:
        J = torch.zeros_like(P)
        out["y"] = _conv(x, kern)
    out.update(dx=dx, decay=-(c * P).real - J.real, freq=-(c * P).imag - J.imag,
               amp=(torch.polar(torch.ones_like(phase), phase) * G).real, phase=-(c * G).imag)
    return out
