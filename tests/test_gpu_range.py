"""Logits and temperatures at the ends of their range: long masked stretches in front of the first allowed token, temperatures
far below one, logits in the billions.  Every row of a batch reads the same logits (row stride 0), so that the kernels see
the shapes of a large batch (one CTA or one warp per logit row) and the oracle only a few rows."""
import math

import numpy as np
import pytest
import torch

import oracle
import paper_2605_02888_b200 as speckv
from paper_2605_02888_b200 import synth, vocab_shard

from parity import compare_step, gpu_batch, mlp_pair, oracle_batch

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
TYPES = {"bf16": torch.bfloat16, "fp32": torch.float32}


def _shared_rows(draft, target, B, T, seed=0):
    """B batch rows over one [G, V] draft and one [G + 1, V] target; the drafted tokens are the draft's first maxima."""
    G = draft.shape[0]
    g = torch.Generator(device=DEV).manual_seed(seed)
    tok = draft.float().argmax(-1).to(torch.int32)
    return dict(draft=draft[None].expand(B, -1, -1), target=target[None].expand(B, -1, -1),
                draft_tokens=tok[None].expand(B, -1).contiguous(), gamma=torch.full((B,), G, dtype=torch.int32, device=DEV),
                temperature=torch.full((B,), T, device=DEV), uniforms=torch.rand(B, G + 1, 2, generator=g, device=DEV),
                comp=torch.zeros(B, 2, device=DEV))


def _oracle(s, rows, om):
    sub = {k: v[torch.as_tensor(rows, device=DEV)] for k, v in s.items()}
    return oracle.step(oracle_batch(sub), sub["comp"].cpu().numpy(), om)


def _check(s, n_shards=0):
    B, G = s["draft_tokens"].shape
    rows = np.unique(np.linspace(0, B - 1, 12).astype(int))
    gm, om = mlp_pair(synth.make_mlp(synth.Workload("r", B=1, gamma_max=G, V=8, seed=1), DEV))
    ref = _oracle(s, rows, om)
    if n_shards:
        out = vocab_shard.step_emulated(gpu_batch(s), n_shards, s["comp"], gm)
    else:
        out = speckv.speckv_step(gpu_batch(s), s["comp"], gm)
        sig = speckv.speckv_signals(gpu_batch(s))
        assert torch.equal(sig["row_status"], out["row_status"])
        for k in ("H", "C"):
            np.testing.assert_allclose(sig[k][rows].cpu().numpy(), ref[k], rtol=1e-5, atol=1e-7, err_msg=k)
    torch.cuda.synchronize()
    compare_step(out, ref, rows=rows)
    return out, ref


# (rows, positions, vocabulary, shards): a lane folds up to 256 elements of a row (short rows, one warp each), 390 to 510
# (the sweep, one CTA per row or per half of an fp32 row), 512 of a slice (one warp per sharded row, two shards)
MASKED = [(256, 4, 8192, 0), (180, 4, 100000, 0), (180, 4, 130999, 0), (560, 4, 32768, 2)]


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("B,G,V,n_shards", MASKED)
@pytest.mark.parametrize("T", [1e-6, 2e-6, 0.8])
def test_masked_stretch_before_the_first_allowed_token(dtype, B, G, V, n_shards, T):
    # constrained decoding: everything but a few tokens is -inf, and those stand at the end of the row
    ninf = float("-inf")
    draft = torch.full((G, V), ninf, device=DEV)
    draft[0, -3:] = torch.tensor([5.0, 5.0, 3.0], device=DEV)      # two tied maxima: H = ln 2 for T near 0
    draft[1, -2] = -1.0                                            # one allowed token
    draft[2, -7:] = 2.0                                            # seven tied maxima
    draft[3, -1] = 5.0                                             # and one in front of the masked stretch
    draft[3, 1] = 5.0
    target = torch.full((G + 1, V), ninf, device=DEV)
    target[:, -7:] = torch.tensor([1.0, 4.0, 4.0, 4.0, 4.0, 4.0, 4.0], device=DEV)
    out, ref = _check(_shared_rows(draft.to(TYPES[dtype]), target.to(TYPES[dtype]), B, T, seed=V), n_shards)
    assert (ref["row_status"] == 0).all()
    if T < 1e-3:
        np.testing.assert_allclose(ref["H"][0], [math.log(2), 0.0, math.log(7), math.log(2)], atol=1e-9)


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("B,G,V,n_shards", [(256, 5, 4096, 0), (2, 5, 40001, 0), (180, 5, 100000, 0), (12, 5, 33000, 3)])
@pytest.mark.parametrize("T,big", [(1.0, 5.0e9), (1.0, 1.0e10), (1.0, 1.0e34), (1e-8, 20.0), (1e-9, 20.0), (1e-9, 0.25)])
def test_draft_logits_far_beyond_the_exponent_range(dtype, B, G, V, n_shards, T, big):
    # logit / T of 1e9 and more: neighbouring values of the exponent's reference are then hundreds apart.  The target stays
    # where include/speckv.h wants it, at a largest |logit| / T below 2^28.
    g = torch.Generator(device=DEV).manual_seed(V)
    dt = TYPES[dtype]
    unit = min(1.0, 1.0e8 * T)
    base = (torch.randn(G + 1, V, generator=g, device=DEV) * unit).clamp(-1.5 * unit, 1.5 * unit)
    draft, target = base[:G].clone(), base.clone()
    draft[0, V - 1] = big                        # met late
    draft[0, V // 2] = big                       # a tie
    draft[1, 3] = big                            # met at once, and a smaller one behind it
    draft[1, V - 2] = big * 0.5
    low = -min(big, 1.0e29)                      # (below -2^100 a logit counts as -inf)
    draft[2] = low                               # flat: H = ln V
    draft[3, : V - 2] = float("-inf")            # masked but for two tokens, the first of which is far below the other
    draft[3, V - 2] = low
    draft[4] = big + base[4]                     # the common offset takes the rest with it (absorbed in part or altogether)
    target[0, V - 1] = 1.5 * unit
    s = _shared_rows(draft.to(dt), target.to(dt), B, T, seed=V)
    out, ref = _check(s, n_shards)
    assert (ref["row_status"] == 0).all()
    assert ref["H"][0, 0] == pytest.approx(math.log(2)) and ref["H"][0, 2] == pytest.approx(math.log(V)) and ref["H"][0, 3] == 0.0


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("B,V,n_shards", [(256, 4096, 0), (3, 40001, 0), (300, 60000, 0), (12, 33000, 3)])
def test_masked_rows_at_temperatures_next_to_zero(dtype, B, V, n_shards):
    # -2^100 / T is beyond fp32 here; draft and target allow a few tokens behind a masked stretch
    G, T = 3, 1e-9
    draft = torch.full((G, V), float("-inf"), device=DEV)
    draft[:, -4:] = torch.tensor([0.25, 0.125, 0.25, -0.25], device=DEV)
    target = torch.full((G + 1, V), float("-inf"), device=DEV)
    target[:, -4:] = torch.tensor([0.25, 0.125, 0.25, 0.25], device=DEV)
    s = _shared_rows(draft.to(TYPES[dtype]), target.to(TYPES[dtype]), B, T, seed=V)
    out, ref = _check(s, n_shards)
    assert (ref["row_status"] == 0).all() and len(set(ref["n_accepted"])) > 1
    u = s["uniforms"][:, :G, 0].contiguous()
    got = speckv.speckv_sample_draft(gpu_batch(s), u)
    assert (got["row_status"] == 0).all()
    assert (got["tokens"] == torch.where(u < 0.5, V - 4, V - 2)).float().mean() > 0.99


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("V,n_shards", [(4096, 0), (40001, 0), (33000, 3)])
@pytest.mark.parametrize("T,level", [(0.9, 0.0), (0.9, 3.0e4), (1e-6, 100.0), (1e-6, 416.0), (1e-6, -416.0), (1e-6, 960.0)])
def test_residual_of_two_tied_tokens(dtype, V, n_shards, T, level):
    # p has two equal maxima and q only the first of them: the residual is the second one alone, whatever the common level
    # of the logits, and its mass of 1/2 must not be taken for an empty one.  Half of the rows reject.  (At T = 1e-6 the
    # normaliser of a row around 416 is 6.0e8 in log2 units and 31 above the nearest fp32 value below it; around 960 it is 63.)
    B, a, b = 40, V // 3, V - 5
    draft = torch.full((1, V), level - 200.0, device=DEV)
    target = draft.expand(2, -1).clone()
    draft[0, a] = level
    target[0, a] = target[0, b] = level
    s = _shared_rows(draft.to(TYPES[dtype]), target.to(TYPES[dtype]), B, T, seed=7)
    s["uniforms"][:, 0, 0] = torch.linspace(0.02, 0.98, B, device=DEV)
    s["uniforms"][:, 0, 1] = torch.linspace(0.03, 0.97, B, device=DEV).flip(0)
    out, ref = _check(s, n_shards)
    rejected = out["n_accepted"] == 0
    assert 10 < int(rejected.sum()) < 30 and (out["out_tokens"][rejected, 0] == b).all()


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("B,V,n_shards", [(256, 4096, 0), (3, 40001, 0), (180, 100000, 0), (12, 33000, 3)])
@pytest.mark.parametrize("T", [1e28, 1e29, 1e30, 1e33])
def test_temperatures_that_flatten_everything(dtype, B, V, n_shards, T):
    # -2^100 / T is small here: what a masked element counts as must still have no weight, and neither may what stands in for a
    # tied maximum that is counted apart or for the elements behind a row's end
    g = torch.Generator(device=DEV).manual_seed(V)
    draft = torch.randn(3, V, generator=g, device=DEV)
    draft[1] = 2.0                                  # every element is the maximum
    draft[2, : V // 2] = float("-inf")
    target = torch.randn(4, V, generator=g, device=DEV)
    s = _shared_rows(draft.to(TYPES[dtype]), target.to(TYPES[dtype]), B, T, seed=V)
    out, ref = _check(s, n_shards)
    assert (ref["row_status"] == 0).all()
    np.testing.assert_allclose(ref["H"][0], [math.log(V), math.log(V), math.log(V - V // 2)], rtol=1e-6)


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("B,V", [(256, 4096), (40, 40001), (300, 60000), (40, 128256)])
@pytest.mark.parametrize("level", [2348810240.0, 2969567232.0, -2164260864.0])
def test_draws_from_rows_far_below_their_reference(dtype, B, V, level):
    # beyond 2^31 in log2 units the fp32 reference of these levels lies 106 to 120 above the row's exponents, and the whole row weighs
    # less than 2^-100: it is drawn from all the same, as a sampled draft and for a bonus token
    scale = np.float32(math.log2(math.e))
    assert 105 < float(np.float32(level) * scale) - float(np.float32(level)) * float(scale) < 121
    G, a, b = 2, V // 3, V - 5
    draft = torch.full((G, V), float("-inf"), device=DEV)
    draft[:, a] = draft[:, b] = level
    s = _shared_rows(draft.to(TYPES[dtype]), draft[:1].expand(G + 1, -1).to(TYPES[dtype]), B, 1.0, seed=3)
    u = torch.linspace(0.02, 0.98, B * G, device=DEV).reshape(G, B).t().contiguous()
    got = speckv.speckv_sample_draft(gpu_batch(s), u)
    assert (got["row_status"] == 0).all() and torch.equal(got["tokens"], torch.where(u < 0.5, a, b).to(torch.int32))
    s["uniforms"][:, :, 0] *= 0.9
    s["uniforms"][:, G, 1] = u[:, 0]
    out = speckv.speckv_verify(gpu_batch(s))
    assert (out["row_status"] == 0).all() and (out["n_accepted"] == G).all()
    assert torch.equal(out["out_tokens"][:, G], torch.where(u[:, 0] < 0.5, a, b).to(torch.int32))
