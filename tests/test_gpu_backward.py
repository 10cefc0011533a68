"""Parity of kda_chunk_bwd (gradients of the prefill operator) with the fp64 backward oracle, through
the C ABI.  Tolerance: relative L2 error 1e-4 per gradient tensor (fp32 FMA arithmetic over at most
a few thousand sequential tokens; stored inputs are exact in both)."""
import numpy as np
import pytest
import torch

import paper_2510_26692_b200 as K
from paper_2510_26692_b200 import inputs
from kda_testlib import Guarded, rel_l2, to_np32

pytestmark = pytest.mark.gpu
TOL = 1e-4
NAMES = ("dq", "dk", "dv", "dlog_alpha", "dbeta", "dS0")


def cotangents(d, seed, dtype):
    T, H, dv = d["v"].shape
    N = d["cu_seqlens"].numel() - 1
    g = torch.Generator().manual_seed(1000 + seed)
    d_o = torch.randn((T, H, dv), generator=g).to(dtype)
    dS_T = torch.randn((N, H, 128, dv), generator=g) * 0.1
    return d_o, dS_T


def run_bwd(d, d_o, dS_T, scale=1.0, dev="cuda:0", want_dS0=True):
    g = {n: (t.to(dev) if isinstance(t, torch.Tensor) else t) for n, t in d.items()}
    T, H, dk = g["k"].shape
    cu = d["cu_seqlens"]
    N = cu.numel() - 1
    dt = K.KDA_BF16 if g["k"].dtype == torch.bfloat16 else K.KDA_F32
    nb = K.kda_chunk_bwd_workspace_bytes(T, N, H)
    ws = Guarded(nb, dev)
    bufs = {"dq": Guarded(T * H * 128 * 4, dev), "dk": Guarded(T * H * 128 * 4, dev),
            "dv": Guarded(T * H * 128 * 4, dev), "dlog_alpha": Guarded(T * H * 128 * 4, dev),
            "dbeta": Guarded(max(T * H * 4, 16), dev), "dS0": Guarded(N * H * 128 * 128 * 4, dev)}
    out = {n: bufs[n].view(torch.float32, (T, H, 128)) for n in ("dq", "dk", "dv", "dlog_alpha")}
    out["dbeta"] = bufs["dbeta"].body[:T * H * 4].view(torch.float32).view(T, H)
    out["dS0"] = bufs["dS0"].view(torch.float32, (N, H, 128, 128))
    for x in out.values():
        x.fill_(float("nan"))
    varlen = N > 1
    K.kda_chunk_bwd(g["q"], g["k"], g["v"], g["log_alpha"], g["beta"], g["S0"],
                    None if d_o is None else d_o.to(dev), None if dS_T is None else dS_T.to(dev),
                    out["dq"], out["dk"], out["dv"], out["dlog_alpha"], out["dbeta"],
                    out["dS0"] if want_dS0 else None, g["cu_seqlens"] if varlen else None,
                    cu if varlen else None, N, T, H, 128, 128, 64, scale, dt, ws.body, nb)
    torch.cuda.synchronize()
    K.kda_check_status(ws.body)
    ws.check("the workspace")
    for n, b_ in bufs.items():
        b_.check(n)
    return out


def oracle_bwd(oracle_mod, d, d_o, dS_T, scale=1.0):
    cu = d["cu_seqlens"].numpy().astype(np.int64)
    return oracle_mod.backward(*(d[n].float().numpy() for n in ("q", "k", "v", "log_alpha", "beta")),
                               d_o=None if d_o is None else d_o.double().numpy(),
                               dS_T=None if dS_T is None else dS_T.double().numpy(),
                               S0=None if d["S0"] is None else d["S0"].double().numpy(),
                               cu_seqlens=cu, scale=scale)


@pytest.mark.parametrize("lens,H,dtype,s0", [([100], 2, torch.float32, 0.0),
                                             ([300], 3, torch.bfloat16, 0.05),
                                             ([64, 1, 200, 0, 130], 2, torch.bfloat16, 0.05),
                                             ([1024], 4, torch.float32, 0.02),
                                             ([3, 0, 9, 64, 65, 1], 1, torch.float32, 0.05),
                                             ([7, 8], 3, torch.bfloat16, 0.0)])
def test_backward_matches_oracle(oracle_mod, lens, H, dtype, s0):
    d = inputs.chunk_inputs(lens, H=H, dtype=dtype, seed=31, s0_std=s0)
    d_o, dS_T = cotangents(d, 31, dtype)
    out = run_bwd(d, d_o, dS_T, scale=0.8)
    ref = oracle_bwd(oracle_mod, d, d_o, dS_T, scale=0.8)
    errs = {n: rel_l2(to_np32(out[n]), ref[n]) for n in NAMES}
    print("bwd", lens, H, dtype, errs)
    for n in NAMES:
        assert torch.isfinite(out[n]).all(), n
        assert errs[n] <= TOL, (n, errs[n])


def test_backward_optional_cotangents_and_determinism(oracle_mod):
    d = inputs.chunk_inputs([200, 70], H=2, dtype=torch.bfloat16, seed=32, s0_std=0.05)
    d_o, dS_T = cotangents(d, 32, torch.bfloat16)
    a = run_bwd(d, d_o, None)
    ref = oracle_bwd(oracle_mod, d, d_o, None)
    for n in NAMES:
        assert rel_l2(to_np32(a[n]), ref[n]) <= TOL, n
    b = run_bwd(d, None, dS_T, want_dS0=False)
    ref = oracle_bwd(oracle_mod, d, None, dS_T)
    for n in NAMES[:-1]:
        assert rel_l2(to_np32(b[n]), ref[n]) <= TOL, n
    a2 = run_bwd(d, d_o, None)
    for n in NAMES:
        assert torch.equal(a[n], a2[n]), n       # fixed summation order: bit-identical runs


def test_backward_argument_errors():
    z = torch.zeros((64, 1, 128), device="cuda:0")
    b = torch.zeros((64, 1), device="cuda:0")
    ws = torch.zeros(1 << 16, dtype=torch.uint8, device="cuda:0")
    with pytest.raises(K.KdaError) as ei:
        K.kda_chunk_bwd(z, z, z, z, b, None, z, None, z.clone(), z.clone(), z.clone(), z.clone(), b.clone(), None,
                        None, None, 1, 64, 1, 128, 128, 64, 1.0, K.KDA_F32, ws)
    assert ei.value.code == 3


@pytest.mark.parametrize("lens,dtype", [([200, 63], torch.float32), ([65, 128, 1], torch.bfloat16)])
def test_backward_fast_decay_heads(oracle_mod, lens, dtype):
    """Heads whose decay leaves the range of the chunk form (log decay below -40 in some chunk) go through
    the token-sequential kernels, the others through the chunk form, in the same call: head 0 stays
    inside, head 1 leaves the range in every chunk, head 2 in one token, head 3 comes close (-38)."""
    d = inputs.chunk_inputs(lens, H=4, dtype=dtype, seed=33, s0_std=0.05)
    la = d["log_alpha"]
    la[:, 1] *= 60.0
    la[40, 2, 7] = -45.0
    la[:, 3] = -38.0 / 64
    d_o, dS_T = cotangents(d, 33, dtype)
    out = run_bwd(d, d_o, dS_T)
    ref = oracle_bwd(oracle_mod, d, d_o, dS_T)
    for n in NAMES:
        x, y = to_np32(out[n]), ref[n]
        for h in range(4):      # (a decay ratio of head 3 carries up to 38 * 2^-24 = 2.3e-6)
            assert rel_l2(x[:, h], y[:, h]) <= TOL, (n, h)


def test_backward_fast_decay_error(oracle_mod):
    """A chunk decays by about e^-37 (the chunk form goes to e^-40): exact exponents leave the products' and sums'
    error, 1.9e-7 on dq; 4.1e-7 with the log decay summed in fp32."""
    d = inputs.chunk_inputs([512], H=4, dtype=torch.float32, seed=33, gate_mean=1.0, s0_std=0.02)
    d_o, dS_T = cotangents(d, 33, torch.float32)
    out, ref = run_bwd(d, d_o, dS_T), oracle_bwd(oracle_mod, d, d_o, dS_T)
    assert rel_l2(to_np32(out["dq"]), ref["dq"]) <= 2.8e-7
    assert rel_l2(to_np32(out["dS0"]), ref["dS0"]) <= 2.2e-7


def test_backward_chains_of_every_length(oracle_mod):
    """Chains of one to six chunks side by side, again and again: the loader's and the products' buffers at every
    phase of their barriers, the same bits each time."""
    lens = [64, 128, 130, 256, 5, 320, 384, 200]
    d = inputs.chunk_inputs(lens, H=5, dtype=torch.bfloat16, seed=34, s0_std=0.02)
    d_o, dS_T = cotangents(d, 34, torch.bfloat16)
    first = run_bwd(d, d_o, dS_T)
    ref = oracle_bwd(oracle_mod, d, d_o, dS_T)
    for n in NAMES:
        assert rel_l2(to_np32(first[n]), ref[n]) <= 1e-5
    for _ in range(10):
        out = run_bwd(d, d_o, dS_T)
        assert all(torch.equal(out[n], first[n]) for n in NAMES)


@pytest.mark.parametrize("lens,H,dtype,harsh", [([9477, 0, 3], 1, torch.bfloat16, None), ([2117, 0, 1, 400], 7, torch.bfloat16, 3),
                                                ([1500, 700], 9, torch.bfloat16, 0), ([1500, 700], 9, torch.float32, 8)])
def test_backward_several_tiles_per_cta(oracle_mod, lens, H, dtype, harsh):
    """More tiles than multiprocessors (150, 294, 315): CTAs go through several, ragged and short ones among them, past the
    tiles of a head that leaves the chunk form in its last chunk, and the last round is not full."""
    d = inputs.chunk_inputs(lens, H=H, dtype=dtype, seed=35, s0_std=0.02)
    if harsh is not None:
        d["log_alpha"][-1, harsh, 5] = -45.0
    d_o, dS_T = cotangents(d, 35, dtype)
    out, ref = run_bwd(d, d_o, dS_T), oracle_bwd(oracle_mod, d, d_o, dS_T)
    for n in NAMES:
        assert rel_l2(to_np32(out[n]), ref[n]) <= 1e-5, n
    again = run_bwd(d, d_o, dS_T)
    assert all(torch.equal(out[n], again[n]) for n in NAMES)


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_calls_queued_without_a_wait(dtype):
    """Launches overlap the end of the call before.  Backward, forward and decode calls queued on one stream and one workspace,
    some on the others' outputs, one with a head out of the chunk form's range: the same bits as with a wait after each."""
    dt = K.KDA_BF16 if dtype == torch.bfloat16 else K.KDA_F32
    T, N, H = 900, 3, 8
    d = [inputs.chunk_inputs([300, 17, 583], H=H, dtype=dtype, seed=s, s0_std=0.02, device="cuda:0") for s in (36, 37)]
    d[1]["log_alpha"][-1, 3, 5] = -45.0
    cot = [[x.cuda() for x in cotangents(d[i], 36 + i, dtype)] for i in range(2)]
    cu = d[0]["cu_seqlens"].cpu()
    cu_dev = cu.cuda()
    nb = max(K.kda_chunk_bwd_workspace_bytes(T, N, H), K.kda_chunk_fwd_workspace_bytes(T, N, H, 128, 128, 64, dt))
    ws = torch.empty(nb, dtype=torch.uint8, device="cuda:0")

    def calls(wait):
        done = []
        after = torch.cuda.synchronize if wait else (lambda: None)

        def backward(x, c, d_o):
            g = {n: torch.full((T, H, 128), float("nan"), device="cuda:0") for n in ("dq", "dk", "dv", "dlog_alpha")}
            g["dbeta"] = torch.full((T, H), float("nan"), device="cuda:0")
            g["dS0"] = torch.full((N, H, 128, 128), float("nan"), device="cuda:0")
            K.kda_chunk_bwd(x["q"], x["k"], x["v"], x["log_alpha"], x["beta"], x["S0"], d_o, c[1], *(g[n] for n in NAMES), cu_dev, cu,
                            N, T, H, 128, 128, 64, 1.0, dt, ws)
            after()
            done.extend(g[n] for n in NAMES)
            return g

        def forward(x, q):
            o, S = torch.empty_like(x["v"]), torch.empty((N, H, 128, 128), device="cuda:0")
            K.kda_chunk_fwd(q, x["k"], x["v"], x["log_alpha"], x["beta"], x["S0"], o, S, cu_dev, cu, N, T, H, 128, 128, 64, 1.0, dt, ws)
            after()
            done.extend((o, S))
            return o, S

        g = backward(d[0], cot[0], cot[0][0])
        o, S = forward(d[1], d[1]["q"])
        backward(d[1], cot[1], o)                       # the forward's outputs, and a head that runs token by token
        o, S = forward(d[0], g["dq"] if dtype == torch.float32 else o)
        x = d[1]
        for t in range(3):                              # the states that have just been written, the row before as q and v
            o1 = torch.empty((N, H, 128), dtype=dtype, device="cuda:0")
            q = x["q"][:N].contiguous() if t == 0 else prev
            K.kda_decode_step(q, x["k"][:N], q, x["log_alpha"][:N], x["beta"][:N], S, None, o1, N, H, 128, 128, 1.0, dt)
            after()
            done.append(o1)
            prev = o1
        backward(d[0], cot[0], cot[0][0])
        torch.cuda.synchronize()
        K.kda_check_status(ws)
        return done

    apart = calls(True)
    assert all(torch.isfinite(x.float()).all() for x in apart)
    for _ in range(5):
        for x, y in zip(calls(False), apart):
            assert torch.equal(x, y)
