"""The draws: a token located from span sums, the span narrowed down by a CTA.  Vocabularies for which a span is one granule
per lane, one level of 8 and of up to 64 parts and two levels deep; draft and target rows that sit differently on the 16-byte
grid; bonus draws (from the sweep's sums), residual draws, draws from p behind an empty residual, draft-side sampling.
Against the oracle under the rules of tests/parity.py, and against a cumulative sum in float64 where the oracle flags."""
import numpy as np
import pytest
import torch

import oracle
import paper_2605_02888_b200 as speckv
from paper_2605_02888_b200 import synth

from parity import compare_step, gpu_batch, mlp_pair, oracle_batch

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
SIZES = [(300, 2, 700), (300, 2, 701), (3, 3, 20001), (40, 2, 151936), (300, 1, 33000), (2, 1, 1100003), (1, 1, 5000003)]


def _workload(B, G, V, dtype, **kw):
    return synth.Workload("d", B=B, gamma_max=G, V=V, dtype=dtype, gamma_mode="ragged", temperature=0.9, sigma_t=1.0,
                          sigma_d=(0.2, 1.0, 2.0), seed=V % 97, **kw)


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("B,G,V", SIZES)
def test_residual_and_bonus_draws(dtype, B, G, V):
    w = _workload(B, G, V, dtype, frac_identical=0.4)
    s = synth.make_step(w, 0, DEV)
    s["uniforms"][: B // 4, :, 1] = 0.0           # first token with weight
    s["uniforms"][B // 4: B // 2, :, 1] = 1.0 - 2.0 ** -24  # last one, or one close to it
    rows = np.arange(B) if B * G * V < 1 << 24 else np.arange(0, B, max(1, B // 24))
    gm, om = mlp_pair(synth.make_mlp(w, DEV))
    out = speckv.speckv_step(gpu_batch(s), s["comp"], gm)
    torch.cuda.synchronize()
    compare_step(out, oracle.step(oracle_batch(s, rows=rows), s["comp"].cpu().numpy()[rows], om), rows=rows)


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("B,G,V", SIZES)
def test_sampled_drafts(dtype, B, G, V):
    w = _workload(B, G, V, dtype)
    s = synth.make_step(w, 0, DEV)
    s["temperature"][::5] = 0.0
    u = torch.rand(B, G, device=DEV)
    rows = np.arange(B) if B * G * V < 1 << 24 else np.arange(0, B, max(1, B // 24))
    tok = speckv.speckv_sample_draft(gpu_batch(s), u)["tokens"].cpu().numpy()[rows]
    ref = oracle.sample_draft(oracle_batch(s, rows=rows), u.cpu().numpy()[rows])
    clear = ref["near"] == 0
    assert (tok[clear] == ref["tokens"][clear]).all() and clear.mean() > 0.9


@pytest.mark.parametrize("dtype,V", [("bf16", 5000), ("fp32", 5001), ("bf16", 300007)])
def test_an_empty_residual_is_drawn_from_p(dtype, V):
    # draft == target and a drafted token without probability: rejected with nothing in the residual
    B = 24
    w = _workload(B, 1, V, dtype, frac_identical=1.0)
    s = synth.make_step(w, 0, DEV)
    s["gamma"][:] = 1
    s["target"][:, 0, 17] = float("-inf")
    s["draft"][:, 0] = s["target"][:, 0]
    s["draft_tokens"][:] = 17
    out = speckv.speckv_verify(gpu_batch(s))
    tok, n = out["out_tokens"][:, 0].cpu().numpy(), out["n_accepted"].cpu().numpy()
    assert (n == 0).all()
    x = s["target"][:, 0].double().cpu().numpy() / 0.9
    p = np.exp(x - x.max(axis=1, keepdims=True))
    cdf = np.cumsum(p, axis=1) / p.sum(axis=1, keepdims=True)
    u = s["uniforms"][:, 0, 1].double().cpu().numpy()
    for b in range(B):  # fp32 weights: the threshold is known to about 1e-6 of the mass (tests/parity.py's window)
        lo, hi = np.searchsorted(cdf[b], u[b] - 1e-6, side="right"), np.searchsorted(cdf[b], u[b] + 1e-6, side="right")
        assert lo <= tok[b] <= hi, (b, lo, tok[b], hi)
