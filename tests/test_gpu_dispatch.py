"""Parity at the sizes where a call changes its kernel variant, against the fp64 oracle."""
import pytest
import torch

import paper_2510_26692_b200 as K
from paper_2510_26692_b200 import inputs
from kda_testlib import TOL, oracle_chunk, rel_l2, run_chunk, to_np32
from test_gpu_layer import oracle_layer, run_layer

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


@pytest.mark.parametrize("lens,H", [([448], 7), ([320], 10), ([70, 1, 64], 3), ([65, 130], 5)])
def test_fp32_prefill_splits(oracle_mod, lens, H):
    """Last and first sizes of tiles in three parts (49 and 50 tiles) and of 8-column chains (9 and 10
    chains).  22-bit operands with fp32 sums: 1e-5."""
    d = inputs.chunk_inputs(lens, H=H, dtype=torch.float32, seed=53, s0_std=0.02)
    o, S = run_chunk(d)
    o_ref, S_ref = oracle_chunk(oracle_mod, d)
    assert rel_l2(to_np32(o), o_ref) <= 1e-5 and rel_l2(to_np32(S), S_ref) <= 1e-5


@pytest.mark.parametrize("lens,H", [([960], 37), ([832], 37), ([896], 38), ([70, 130], 37), ([1] * 256 + [90], 1)])
def test_bf16_schedules(oracle_mod, lens, H):
    """Fused kernel and two kernels near the line between them, and more sequences than the table of
    lengths holds.  Operands rounded to bf16: TOL."""
    d = inputs.chunk_inputs(lens, H=H, dtype=torch.bfloat16, seed=54, s0_std=0.02)
    o, S = run_chunk(d)
    o_ref, S_ref = oracle_chunk(oracle_mod, d)
    assert rel_l2(to_np32(o), o_ref) <= TOL[K.KDA_BF16] and rel_l2(to_np32(S), S_ref) <= TOL[K.KDA_BF16]


@pytest.mark.parametrize("lens,H,out", [([4100], 3, True), ([4033], 3, False), ([5000, 70, 0, 2000], 1, True),
                                        ([6000, 64, 3000], 2, False)])
def test_bf16_segments(oracle_mod, lens, H, out):
    """Chains cut into segments, the last ones short or empty: within TOL of the oracle and no further
    from it than the uncut chains but for the rounding of other operands (a tenth)."""
    d = inputs.chunk_inputs(lens, H=H, dtype=torch.bfloat16, seed=55, s0_std=0.02)
    o_ref, S_ref = oracle_chunk(oracle_mod, d)
    err = []
    for mode in (0, 1):
        K.kda_set_chunk_path(mode)
        try:
            before = K.kda_launch_count()
            o, S = run_chunk(d, want_o=out)
            launches = K.kda_launch_count() - before
        finally:
            K.kda_set_chunk_path(0)
        err.append((launches, rel_l2(to_np32(o), o_ref) if out else 0.0, rel_l2(to_np32(S), S_ref)))
    (n0, eo0, es0), (n1, eo1, es1) = err
    assert n0 == n1 + (2 if out else 1)       # it was cut
    assert eo0 <= min(TOL[K.KDA_BF16], 1.1 * eo1) and es0 <= min(TOL[K.KDA_BF16], 1.1 * es1)


@pytest.mark.parametrize("T,H,out,launches", [(1024, 32, False, 2), (960, 37, False, 2), (4096, 32, True, 1), (3072, 28, True, 1),
                                              (10240, 34, True, 4), (6144, 48, True, 2), (3072, 24, False, 3)])
def test_bf16_schedule_near_the_lines(T, H, out, launches):
    """The way a call takes near the lines between two kernels, the fused kernel (1 launch) and segments (with outputs 2 more
    than two kernels, else 1): the fastest measured, by 6 to 20 per cent.  Results as on the two kernels but for the rounding
    of other operands to bf16 (TOL)."""
    d = inputs.chunk_inputs([T], H=H, dtype=torch.bfloat16, seed=58, s0_std=0.02, device="cuda:0")
    got = {}
    for mode in (0, 1):
        K.kda_set_chunk_path(mode)
        try:
            before = K.kda_launch_count()
            got[mode] = run_chunk(d, want_o=out) + (K.kda_launch_count() - before,)
        finally:
            K.kda_set_chunk_path(0)
    assert got[1][2] == 2 and got[0][2] == launches
    for x, y in zip(got[0][:2], got[1][:2]):
        assert x is None and y is None or rel_l2(to_np32(x), to_np32(y)) <= TOL[K.KDA_BF16]


@pytest.mark.parametrize("lens,H", [([300, 70], 18), ([300, 70], 19), ([4100], 3)])
def test_layer_output_rows(oracle_mod, lens, H):
    """Output stage from fp32 rows (up to 37 chains) and from bf16 rows, chains whole and in segments:
    bf16 operands and output, TOL."""
    d = inputs.layer_inputs(lens, H=H, seed=56, s0_std=0.02)
    y, S = run_layer(d, 128 ** -0.5)
    y_ref, S_ref, _ = oracle_layer(oracle_mod, d, 128 ** -0.5)
    assert rel_l2(to_np32(y), y_ref) <= TOL[K.KDA_BF16] and rel_l2(to_np32(S), S_ref) <= TOL[K.KDA_BF16]


@pytest.mark.parametrize("lens,H", [([1024], 32), ([1024], 38)])
def test_bf16_one_rounding_of_q(oracle_mod, lens, H):
    """Q is rounded to bf16 once: Aqk and Q S use the same numbers (fused kernel and two kernels).  At a decay of
    sigmoid(6) a token the error of o is 4.82e-3 by that arithmetic in fp64 with rounded operands; 4.87e-3 with the
    two products' Q rounded apart."""
    d = inputs.chunk_inputs(lens, H=H, dtype=torch.bfloat16, seed=57, gate_mean=6.0, s0_std=0.02)
    o, _ = run_chunk(d)
    o_ref, _ = oracle_chunk(oracle_mod, d)
    assert rel_l2(to_np32(o), o_ref) <= 4.85e-3


@pytest.mark.parametrize("H", [2, 37])
def test_fp32_prefill_fast_decay(oracle_mod, H):
    """Decay of about e^-84 a chunk: the exponents are exact, so the error stays that of the products and sums (2.0e-7
    at slow decay, plus that of entries far below the largest); 7.2e-7 and 9.8e-7 with the log decay summed in fp32."""
    d = inputs.chunk_inputs([300], H=H, dtype=torch.float32, seed=58, gate_mean=-1.0, s0_std=0.02)
    o, S = run_chunk(d)
    o_ref, S_ref = oracle_chunk(oracle_mod, d)
    assert rel_l2(to_np32(o), o_ref) <= 4e-7 and rel_l2(to_np32(S), S_ref) <= 3e-7


@pytest.mark.parametrize("tiles,H,out", [(2, 5, True), (7, 5, True), (40, 5, False), (150, 5, True), (900, 32, True), (900, 32, False)])
def test_fused_hand_over(tiles, H, out):
    """The fused kernel against the two kernels, the same bits each time, with rings from two tiles in all to four
    per engine: a tile read before it is written, or written over before it is read, would show."""
    d = inputs.chunk_inputs([700, 130, 64, 1, 0, 950], H=H, dtype=torch.bfloat16, seed=59, s0_std=0.02)
    small = K.kda_chunk_fwd_min_workspace_bytes(1845, 6, H)
    tile = small - 256 >> 1
    try:
        K.kda_set_chunk_path(1)
        o1, S1 = run_chunk(d, want_o=out)
        K.kda_set_chunk_path(2)
        for _ in range(12):
            o2, S2 = run_chunk(d, want_o=out, workspace_bytes=small + (tiles - 2) * tile)
            assert torch.equal(S1, S2) and (not out or torch.equal(o1, o2))
    finally:
        K.kda_set_chunk_path(0)


@pytest.mark.parametrize("lens,fused", [([4000] + [600] * 6, True), ([1100] * 7, False)])
def test_uneven_batches_take_the_faster_schedule(oracle_mod, lens, fused):
    """More chains (56) than clusters: one launch where a few long chains set the time, three kernels (chunk table, tiles,
    chains) where all are alike.  Operands rounded to bf16: TOL."""
    d = inputs.chunk_inputs(lens, H=8, dtype=torch.bfloat16, seed=60, s0_std=0.02)
    before = K.kda_launch_count()
    o, S = run_chunk(d)
    assert K.kda_launch_count() - before == (1 if fused else 3)
    o_ref, S_ref = oracle_chunk(oracle_mod, d)
    assert rel_l2(to_np32(o), o_ref) <= TOL[K.KDA_BF16] and rel_l2(to_np32(S), S_ref) <= TOL[K.KDA_BF16]


def test_bf16_segments_in_passes(oracle_mod):
    """The final state of one sequence with a workspace for 320 chunks of 323: cut into segments twice, the state of the
    first pass entering the second, whose 3 chunks are fewer than the segments.  No further from the oracle than the
    uncut chains but for other roundings (a tenth)."""
    H, T = 16, 323 * 64 - 30
    d = inputs.chunk_inputs([T], H=H, dtype=torch.bfloat16, seed=66, s0_std=0.02)
    tile = (K.kda_chunk_fwd_min_workspace_bytes(T, 1, H) - 256) // 2
    row = H * tile
    fixed = K.kda_layer_fwd_min_workspace_bytes(T, 1, H) - row
    nbytes = fixed + 320 * row + 148 * 65536 + 256
    assert nbytes < K.kda_chunk_fwd_workspace_bytes(T, 1, H)
    _, S_ref = oracle_chunk(oracle_mod, d, want_o=False)
    before = K.kda_launch_count()
    _, S = run_chunk(d, want_o=False, workspace_bytes=nbytes)
    assert K.kda_launch_count() - before == 6          # tiles, maps, states: twice
    K.kda_set_chunk_path(1)
    try:
        _, S1 = run_chunk(d, want_o=False)
    finally:
        K.kda_set_chunk_path(0)
    err = rel_l2(to_np32(S), S_ref)
    assert err <= TOL[K.KDA_BF16] and err <= 1.1 * rel_l2(to_np32(S1), S_ref)


@pytest.mark.parametrize("out", [True, False])
@pytest.mark.parametrize("lens,H", [([4100], 3), ([5000, 4000], 8)])
def test_bf16_long_chains_in_place(oracle_mod, lens, H, out):
    """S_T over S0 where chains are cut for the state alone, and may not be with outputs: the last segment would write
    the state that the first may still have to read."""
    d = inputs.chunk_inputs(lens, H=H, dtype=torch.bfloat16, seed=67, s0_std=0.3, device="cuda:0")
    T, N, cu = sum(lens), len(lens), d["cu_seqlens"]
    S = d["S0"].clone()
    o = torch.full_like(d["v"], float("nan")) if out else None
    ws = torch.empty(K.kda_chunk_fwd_workspace_bytes(T, N, H), dtype=torch.uint8, device="cuda:0")
    before = K.kda_launch_count()
    K.kda_chunk_fwd(d["q"] if out else None, d["k"], d["v"], d["log_alpha"], d["beta"], S, o, S, cu.cuda() if N > 1 else None,
                    cu.cpu() if N > 1 else None, N, T, H, 128, 128, 64, 1.0, K.KDA_BF16, ws)
    torch.cuda.synchronize()
    launches = K.kda_launch_count() - before
    if out:
        assert launches <= 2 + (N > 1)                  # not cut
    else:
        assert launches == 3 + (N > 1)                  # (chunk table,) tiles, maps, states
    o_ref, S_ref = oracle_chunk(oracle_mod, d, want_o=out)
    assert rel_l2(to_np32(S), S_ref) <= TOL[K.KDA_BF16]
    assert not out or rel_l2(to_np32(o), o_ref) <= TOL[K.KDA_BF16]
