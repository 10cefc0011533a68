"""The work that users of this library have it do, as cases that can be timed and compared.

Kimi Delta Attention is used in three places: prompts are prefilled (one prompt, many packed
prompts, one very long context), tokens are generated (one or a few per sequence and call), and the
operator is trained (its backward pass).  A case is one call of a public entry point with the
buffers that a serving or training program has at hand; ``draw`` gives further cases of the same
ranges.  ``dk = dv = 128`` and chunks of 64 tokens throughout (the supported shape).

Keys of a case: ``op``; ``H`` heads; ``dtype`` of q, k, v, o; ``seqs`` sequences whose lengths lie in
``lo`` .. ``hi`` (drawn from the number ``lens``; equal bounds give one fixed length); ``tokens`` per
sequence of a decode call; ``s0`` whether initial states are given; ``gate`` the mean of the decay's
logit; ``out`` whether the outputs are wanted besides the final states; ``slots`` whether decode
states are addressed through a slot table.
"""
from __future__ import annotations

import torch

import paper_2510_26692_b200 as K
from paper_2510_26692_b200 import inputs

D = 128
STATE = D * D * 4
L2_EPS, RMS_EPS = 1e-6, 1e-5
DEV = "cuda"


def listed():
    return [
        # One user's generation loop: one sequence, one token, one layer of a 32-head model.
        dict(name="decode 1x32", op="decode", seqs=1, H=32, dtype="bf16", tokens=1, slots=False),
        # The decode step of a full serving batch.
        dict(name="decode 256x32", op="decode", seqs=256, H=32, dtype="bf16", tokens=1, slots=False),
        # A partly filled batch whose states live in a paged cache, with the layer's norms and gates.
        dict(name="layer decode 37x32 slots", op="layer_decode", seqs=37, H=32, dtype="bf16", tokens=1, slots=True),
        # Verification of speculated tokens: four per sequence.
        dict(name="decode multi 64x32 4 tok", op="decode", seqs=64, H=32, dtype="bf16", tokens=4, slots=False),
        # Prefill in full precision (checks of a model, small research models).
        dict(name="prefill fp32 256 H2", op="prefill", seqs=1, lo=256, hi=256, lens=0, H=2, dtype="fp32", s0=False,
             gate=4.0, out=True),
        # A few short prompts of odd lengths that arrive together.
        dict(name="prefill 5 short prompts", op="prefill", seqs=5, lo=17, hi=300, lens=11, H=32, dtype="bf16", s0=False,
             gate=4.0, out=True),
        # One ordinary prompt segment that continues from a cached state.
        dict(name="prefill 4096", op="prefill", seqs=1, lo=4096, hi=4096, lens=0, H=32, dtype="bf16", s0=True, gate=4.0,
             out=True),
        # A large packed batch of uneven prompts.
        dict(name="prefill packed 16", op="prefill", seqs=16, lo=512, hi=16384, lens=2, H=32, dtype="bf16", s0=True,
             gate=4.0, out=True),
        # A million-token context read in for its final state, slow decay.
        dict(name="prefill 1Mi state", op="prefill", seqs=1, lo=1 << 20, hi=1 << 20, lens=0, H=32, dtype="bf16", s0=True,
             gate=6.0, out=False),
        # The layer's whole operator (norms, decay function, output gate) on three ragged prompts.
        dict(name="layer 3 prompts", op="layer", seqs=3, lo=900, hi=4100, lens=5, H=32, dtype="bf16", s0=True, gate=4.0,
             out=True),
        # A training step's backward pass, sequence length and heads of the ordinary prefill.
        dict(name="backward 4096", op="backward", seqs=1, lo=4096, hi=4096, lens=0, H=32, dtype="bf16", s0=True, gate=4.0,
             out=True),
        # Backward over a packed batch of short uneven sequences in full precision.
        dict(name="backward fp32 packed 6", op="backward", seqs=6, lo=40, hi=700, lens=3, H=8, dtype="fp32", s0=False,
             gate=4.0, out=True),
    ]


def _spread(rng, lo, hi):
    """A whole number between lo and hi, spread over the logarithm."""
    return min(hi, max(lo, int(round(lo * (hi / lo) ** rng.random()))))


def _packed(rng, most):
    """seqs, lo, hi, lens of a batch of at most ``most`` tokens."""
    seqs = rng.choice((1, 1, 2, 3, 4, 7, 8, 16))
    hi = _spread(rng, 17, most // seqs)
    lo = hi if seqs == 1 else max(1, int(hi * rng.uniform(0.05, 0.9)))
    return dict(seqs=seqs, lo=lo, hi=hi, lens=rng.randrange(1000))


def draw(rng):
    op = rng.choice(("decode", "decode", "multi", "layer_decode", "prefill", "prefill", "fp32", "long", "layer", "backward",
                     "backward"))
    if op == "decode":
        return dict(op="decode", seqs=_spread(rng, 1, 256), H=rng.choice((8, 16, 32)), tokens=1,
                    dtype=rng.choice(("bf16", "bf16", "fp32")), slots=rng.random() < 0.5)
    if op == "multi":
        return dict(op="decode", seqs=_spread(rng, 1, 128), H=rng.choice((8, 16, 32)), tokens=rng.randint(2, 8), dtype="bf16",
                    slots=rng.random() < 0.5)
    if op == "layer_decode":
        return dict(op="layer_decode", seqs=_spread(rng, 1, 256), H=rng.choice((8, 16, 32)), tokens=1, dtype="bf16",
                    slots=rng.random() < 0.5)
    if op == "prefill":
        return dict(op="prefill", H=rng.choice((8, 16, 32)), dtype="bf16", s0=rng.random() < 0.5, gate=4.0, out=True,
                    **_packed(rng, 131072))
    if op == "fp32":
        return dict(op="prefill", H=rng.choice((2, 4, 8)), dtype="fp32", s0=rng.random() < 0.5, gate=4.0, out=True,
                    **_packed(rng, 2048))
    if op == "long":
        n = _spread(rng, 1 << 16, 1 << 20)
        return dict(op="prefill", seqs=1, lo=n, hi=n, lens=0, H=rng.choice((16, 32)), dtype="bf16", s0=True, gate=6.0,
                    out=False)
    if op == "layer":
        return dict(op="layer", H=rng.choice((8, 16, 32)), dtype="bf16", s0=rng.random() < 0.5, gate=4.0, out=True,
                    **_packed(rng, 32768))
    return dict(op="backward", H=rng.choice((4, 8, 16, 32)), dtype=rng.choice(("bf16", "bf16", "fp32")),
                s0=rng.random() < 0.5, gate=4.0, out=True, **_packed(rng, 8192))


def _lengths(c):
    if c["lo"] == c["hi"]:
        return [c["lo"]] * c["seqs"]
    return inputs.varlen_lengths(c["seqs"], c["lo"], c["hi"], c["lens"])


def _types(c):
    return (torch.bfloat16, K.KDA_BF16) if c["dtype"] == "bf16" else (torch.float32, K.KDA_F32)


def _empty(*shape, dtype=torch.float32):
    return torch.empty(shape, dtype=dtype, device=DEV)


def _batch(c, st):
    """What every call over packed sequences needs besides its tensors."""
    lens = _lengths(c)
    st.update(N=c["seqs"], T=sum(lens), cu_dev=None, cu_host=None)
    if c["seqs"] > 1:
        st["cu_host"] = inputs.cu_seqlens_of(lens)
        st["cu_dev"] = st["cu_host"].to(DEV)
    return lens


def prepare(case, seed):
    c = case
    H, (et, dt) = c["H"], _types(c)
    st = dict(case=c, H=H, dt=dt)
    if c["op"] == "decode":
        N, n_tok = c["seqs"], c["tokens"]
        d = inputs.decode_inputs(N, H, n_tok, dtype=et, seed=seed, device=DEV)
        for n in ("q", "k", "v", "log_alpha", "beta"):      # [tokens, N, ...] -> [N, tokens, ...]
            st[n] = d[n][0] if n_tok == 1 else d[n].transpose(0, 1).contiguous()
        st.update(S=d["S"], o=torch.empty_like(st["v"]), N=N)
    elif c["op"] == "layer_decode":
        N = c["seqs"]
        st.update(inputs.layer_inputs([N], H, seed=seed, device=DEV))
        st.update(S=inputs.decode_inputs(N, H, 1, seed=seed, device=DEV)["S"], y=torch.empty_like(st["v"]), N=N)
    if c["op"] in ("decode", "layer_decode"):
        st["slot"] = None
        if c["slots"]:                                      # a cache with room for half as many sequences again
            N = c["seqs"]
            n_slots = N + (N + 1) // 2
            S = torch.zeros((n_slots, H, D, D), device=DEV)
            g = torch.Generator(device="cpu")
            g.manual_seed(int(seed))
            slot = torch.randperm(n_slots, generator=g)[:N].to(DEV)
            S[slot] = st["S"]
            st.update(S=S, slot=slot.to(torch.int32))
        return st

    lens = _batch(c, st)
    N, T = st["N"], st["T"]
    s0 = 0.02 if c["s0"] else 0.0
    st["S_T"] = _empty(N, H, D, D)
    if c["op"] == "layer":
        st.update(inputs.layer_inputs(lens, H, seed=seed, gate_mean=c["gate"], s0_std=s0, device=DEV))
        st["y"] = torch.empty_like(st["v"])
        ws = K.kda_layer_fwd_workspace_bytes(T, N, H)
    elif c["op"] == "prefill":
        if N == 1 and dt == K.KDA_BF16:                     # drawn slab by slab: no large temporaries
            st.update(inputs.chunk_inputs_slabbed(T, H, seed=seed, gate_mean=c["gate"], s0_std=s0, device=DEV,
                                                  want_q=c["out"]))
        else:
            st.update(inputs.chunk_inputs(lens, H, dtype=et, seed=seed, gate_mean=c["gate"], s0_std=s0, device=DEV))
        st["o"] = torch.empty_like(st["v"]) if c["out"] else None
        ws = K.kda_chunk_fwd_workspace_bytes(T, N, H, D, D, 64, dt)
    else:
        st.update(inputs.chunk_inputs(lens, H, dtype=et, seed=seed, gate_mean=c["gate"], s0_std=s0, device=DEV))
        g = torch.Generator(device=DEV)
        g.manual_seed(int(seed) * 16 + 15)
        st["d_o"] = torch.randn((T, H, D), generator=g, device=DEV).to(et)
        st["dS_T"] = torch.randn((N, H, D, D), generator=g, device=DEV) * 0.1 if c["s0"] else None
        st.update(dq=_empty(T, H, D), dk=_empty(T, H, D), dv=_empty(T, H, D), dg=_empty(T, H, D), db=_empty(T, H),
                  dS0=_empty(N, H, D, D) if c["s0"] else None)
        ws = K.kda_chunk_bwd_workspace_bytes(T, N, H)
    st["ws"] = torch.empty(ws, dtype=torch.uint8, device=DEV)
    return st


def run(state):
    s = state
    c, H = s["case"], s["H"]
    if c["op"] == "decode":
        if c["tokens"] == 1:
            K.kda_decode_step(s["q"], s["k"], s["v"], s["log_alpha"], s["beta"], s["S"], s["slot"], s["o"], s["N"], H, D, D,
                              1.0, s["dt"])
        else:
            K.kda_decode_multi(s["q"], s["k"], s["v"], s["log_alpha"], s["beta"], s["S"], s["slot"], s["o"], s["N"],
                               c["tokens"], H, D, D, 1.0, s["dt"])
        return s["o"], s["S"]
    if c["op"] == "layer_decode":
        K.kda_layer_decode_step(s["q_c"], s["k_c"], s["v"], s["g_a"], s["b_pre"], s["g_o"], s["A_log"], s["dt_bias"], s["w"],
                                L2_EPS, RMS_EPS, s["S"], s["slot"], s["y"], s["N"], H, D, D, D ** -0.5)
        return s["y"], s["S"]
    if c["op"] == "layer":
        K.kda_layer_fwd(s["q_c"], s["k_c"], s["v"], s["g_a"], s["b_pre"], s["g_o"], s["A_log"], s["dt_bias"], s["w"], L2_EPS,
                        RMS_EPS, s["S0"], s["y"], s["S_T"], s["cu_dev"], s["cu_host"], s["N"], s["T"], H, D, D, 64,
                        D ** -0.5, s["ws"])
        return s["y"], s["S_T"]
    if c["op"] == "prefill":
        K.kda_chunk_fwd(s["q"] if c["out"] else None, s["k"], s["v"], s["log_alpha"], s["beta"], s["S0"], s["o"], s["S_T"],
                        s["cu_dev"], s["cu_host"], s["N"], s["T"], H, D, D, 64, 1.0, s["dt"], s["ws"])
        return (s["o"], s["S_T"]) if c["out"] else s["S_T"]
    K.kda_chunk_bwd(s["q"], s["k"], s["v"], s["log_alpha"], s["beta"], s["S0"], s["d_o"], s["dS_T"], s["dq"], s["dk"],
                    s["dv"], s["dg"], s["db"], s["dS0"], s["cu_dev"], s["cu_host"], s["N"], s["T"], H, D, D, 64, 1.0,
                    s["dt"], s["ws"])
    return {n: s[n] for n in ("dq", "dk", "dv", "dg", "db", "dS0") if s[n] is not None}


def work(case):
    """Bytes: every input once in, every output once out.  Flops: for a decode token the recurrence
    (decay, two contractions with the state, one rank-one update); for a chunked token the chunkwise
    form's 6 d^2 + 3 C d + C^2 per head; for the backward pass three times that (the forward again
    and two products for each of its products)."""
    c = case
    es = 2 if c["dtype"] == "bf16" else 4
    H = c["H"]
    if c["op"] in ("decode", "layer_decode"):
        n = c["seqs"] * H * c["tokens"]
        row = D * 4 * es + D * 4 + 4 if c["op"] == "decode" else D * 6 * es + 4
        return dict(bytes=c["seqs"] * H * 2 * STATE + n * row, flops=n * 7 * D * D)
    T, N = sum(_lengths(c)), c["seqs"]
    n = T * H
    flops = 6 * D * D + 3 * 64 * D + 64 * 64
    states = N * H * STATE * (2 if c["s0"] else 1)
    if c["op"] == "layer":
        return dict(bytes=n * (6 * D * 2 + 4) + states, flops=n * flops)
    if c["op"] == "prefill":
        if c["out"]:
            return dict(bytes=n * (4 * D * es + D * 4 + 4) + states, flops=n * flops)
        return dict(bytes=n * (2 * D * es + D * 4 + 4) + states, flops=n * (4 * D * D + 2 * 64 * D + 64 * 64))
    states = N * H * STATE * (3 if c["s0"] else 0)
    return dict(bytes=n * (4 * D * es + D * 4 + 4 + 4 * D * 4 + 4) + states, flops=n * 3 * flops)


def tolerance(case):
    """fp32 arithmetic throughout (fp32 prefill; the backward pass whatever the storage of q, k, v;
    fp32 decode): rounding of 32-bit sums.  Otherwise bf16 outputs, or bf16 tensor-core operands."""
    if case["dtype"] == "fp32" or case["op"] == "backward":
        return {"rel": 1e-5}
    return {"rel": 1e-2}
