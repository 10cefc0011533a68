"""What a NaN or an infinity in one token does: everything that Eq. 1 makes non-finite (the fp64 oracle on the
same inputs) is not finite in the outputs either, and the other head is untouched."""
import numpy as np
import pytest
import torch

import paper_2510_26692_b200 as K
from paper_2510_26692_b200 import inputs
from kda_testlib import oracle_chunk, run_chunk, to_np32
from test_gpu_backward import cotangents, oracle_bwd, run_bwd

pytestmark = pytest.mark.gpu
NAN, INF = float("nan"), float("inf")


def spoiled(d, what, token, value):
    """The inputs with one element of head 0 replaced."""
    d = dict(d)
    d[what] = d[what].clone()
    if what == "beta":
        d[what][token, 0] = value
    else:
        d[what][token, 0, 5] = value
    return d


@pytest.mark.parametrize("what,value", [("q", NAN), ("k", NAN), ("v", NAN), ("beta", NAN), ("log_alpha", NAN),
                                        ("q", INF), ("k", INF), ("v", INF), ("beta", INF)])
def test_fp32_prefill_keeps_non_finite(oracle_mod, what, value):
    d = spoiled(inputs.chunk_inputs([200], H=2, dtype=torch.float32, seed=61, s0_std=0.02), what, 100, value)
    o, S = run_chunk(d)
    o_ref, S_ref = oracle_chunk(oracle_mod, d)
    bad_o, bad_S = ~np.isfinite(to_np32(o)), ~np.isfinite(to_np32(S))
    assert bad_o[~np.isfinite(o_ref)].all() and bad_S[~np.isfinite(S_ref)].all()
    assert not bad_o[:64].any() and not bad_o[:, 1].any() and not bad_S[:, 1].any()


@pytest.mark.parametrize("token", [0, 100, 127])
@pytest.mark.parametrize("H", [2, 37])
@pytest.mark.parametrize("what,value", [("q", NAN), ("k", NAN), ("v", NAN), ("beta", NAN), ("log_alpha", NAN),
                                        ("k", INF), ("v", INF)])
def test_fp32_prefill_non_finite_is_causal(oracle_mod, what, value, H, token):
    """A tile in three CTAs (2 heads) and in one (37): what the recurrence leaves finite, the earlier tokens of
    the same chunk among it, is finite and right (22-bit operands, fp32 sums: 1e-5)."""
    d = spoiled(inputs.chunk_inputs([200], H=H, dtype=torch.float32, seed=63, s0_std=0.02), what, token, value)
    o, S = (to_np32(x) for x in run_chunk(d))
    o_ref, S_ref = oracle_chunk(oracle_mod, d)
    for x, ref in ((o, o_ref), (S, S_ref)):
        assert (np.isfinite(x) == np.isfinite(ref)).all()
        ok = np.isfinite(ref)
        assert np.linalg.norm(x[ok] - ref[ok]) <= 1e-5 * np.linalg.norm(ref[ok])


@pytest.mark.parametrize("what,value", [("k", NAN), ("v", NAN), ("log_alpha", NAN), ("v", INF)])
def test_segments_keep_non_finite(oracle_mod, what, value):
    """Chains that are cut into segments: the state over a border is as non-finite as the one before it."""
    d = spoiled(inputs.chunk_inputs([4100], H=2, dtype=torch.bfloat16, seed=62), what, 700, value)
    o, S = run_chunk(d)
    o_ref, S_ref = oracle_chunk(oracle_mod, d)
    bad_o, bad_S = ~np.isfinite(to_np32(o)), ~np.isfinite(to_np32(S))
    assert bad_o[~np.isfinite(o_ref)].all() and bad_S[~np.isfinite(S_ref)].all()
    assert not bad_o[:640].any() and not bad_o[:, 1].any() and not bad_S[:, 1].any()
    _, S = run_chunk(d, want_o=False)
    assert (~np.isfinite(to_np32(S)))[~np.isfinite(S_ref)].all()


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("what,value", [("q", NAN), ("k", NAN), ("v", NAN), ("beta", NAN), ("d_o", NAN), ("k", INF),
                                        ("v", INF), ("d_o", INF)])
def test_backward_non_finite(oracle_mod, what, value, dtype):
    """Gradients are finite where the adjoint of the recurrence is, tokens of the same chunk among them, and right
    there (fp32 arithmetic: 1e-5)."""
    d = inputs.chunk_inputs([200], H=2, dtype=dtype, seed=64, s0_std=0.02)
    d["d_o"], dS_T = cotangents(d, 65, dtype)
    d = spoiled(d, what, 100, value)
    got, ref = run_bwd(d, d["d_o"], dS_T), oracle_bwd(oracle_mod, d, d["d_o"], dS_T)
    for n, x in got.items():
        x, ok = to_np32(x), np.isfinite(ref[n])
        assert (np.isfinite(x) == ok).all(), n
        assert np.linalg.norm(x[ok] - ref[n][ok]) <= 1e-5 * np.linalg.norm(ref[n][ok]), n
