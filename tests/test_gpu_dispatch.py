"""Parity at the sizes where a call changes its kernel variant, against the fp64 oracle."""
import pytest
import torch

import paper_2510_26692_b200 as K
from paper_2510_26692_b200 import inputs
from kda_testlib import rel_l2, to_np32

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("items", [1, 222, 223, 296, 297, 5920, 5921])
def test_decode_column_slices(oracle_mod, items, dtype):
    """Half and whole states per CTA: the state within fp32 rounding of its 128-term sums (1e-6), o
    within that or its bf16 rounding (2^-9 relative); two steps that follow each other without a wait."""
    d = inputs.decode_inputs(items, 1, 2, dtype=dtype, seed=51)
    dt = K.KDA_BF16 if dtype == torch.bfloat16 else K.KDA_F32
    g = {n: x.to("cuda:0") for n, x in d.items()}
    o = torch.full((2, items, 1, 128), float("nan"), dtype=dtype, device="cuda:0")
    for t in range(2):
        K.kda_decode_step(g["q"][t], g["k"][t], g["v"][t], g["log_alpha"][t], g["beta"][t].clone(), g["S"], None, o[t],
                          items, 1, 128, 128, 0.7, dt)
    torch.cuda.synchronize()
    S = d["S"].double().numpy().copy()
    for t in range(2):
        ref = oracle_mod.decode_step(*(to_np32(d[n][t]) for n in ("q", "k", "v", "log_alpha", "beta")), S, scale=0.7)
        assert rel_l2(to_np32(o[t]), ref) <= (2e-6 if dtype == torch.float32 else 2.0 ** -9)
    assert rel_l2(to_np32(g["S"]), S) <= 1e-6


def test_binding_takes_what_it_took():
    """Arguments outside the native marshalling's plain kind still work or raise as before: numbers that
    are not exactly int / float, an explicit stream, wrong device, type and layout."""
    d = inputs.decode_inputs(3, 2, 1, seed=52, device="cuda:0")
    a = [d[n][0] for n in ("q", "k", "v", "log_alpha", "beta")]
    o = torch.empty_like(a[2])
    outs = []
    for scale, n, stream in ((1.0, 3, None), (1, torch.tensor(3).item(), torch.cuda.current_stream()), (True, 3, None)):
        S = d["S"].clone()
        K.kda_decode_step(*a, S, None, o, n, 2, 128, 128, scale, K.KDA_BF16, stream=stream)
        outs.append((o.clone(), S))
    for x, S in outs[1:]:
        assert torch.equal(x, outs[0][0]) and torch.equal(S, outs[0][1])
    with pytest.raises(ValueError, match="live on"):
        K.kda_decode_step(a[0].cpu(), *a[1:], d["S"], None, o, 3, 2, 128, 128, 1.0, K.KDA_BF16)
    with pytest.raises(TypeError, match="must be"):
        K.kda_decode_step(a[0].float(), *a[1:], d["S"], None, o, 3, 2, 128, 128, 1.0, K.KDA_BF16)
    with pytest.raises(ValueError, match="contiguous"):
        K.kda_decode_step(a[0].transpose(0, 1), *a[1:], d["S"], None, o, 3, 2, 128, 128, 1.0, K.KDA_BF16)
    with pytest.raises(K.KdaError) as ei:
        K.kda_decode_step(*a, d["S"], None, None, 3, 2, 128, 128, 1.0, K.KDA_BF16)
    assert ei.value.code == 1
