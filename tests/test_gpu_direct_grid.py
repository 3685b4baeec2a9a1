"""Small batches: the sweep's CTAs find their work from gamma and the temperatures themselves, and a rejected row is drawn from by
CTAs of its own that wait for the row's record and for one another's sums.  Up to 256 batch rows and the next size, draws by 1 to 16
CTAs, rows off the 16-byte grid, rows that are flagged and have no logit row in use; and waits that run out at once."""
import numpy as np
import pytest
import torch

import oracle
import paper_2605_02888_b200 as speckv
from paper_2605_02888_b200 import binding, synth

from parity import compare_step, gpu_batch, mlp_pair, oracle_batch, plan_of

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _step(B, G, V, dtype):
    w = synth.Workload("direct", B=B, gamma_max=G, V=V, dtype=dtype, gamma_mode="ragged", temperature=0.9, sigma_t=1.0,
                       sigma_d=(0.3, 1.0, 2.0), frac_identical=0.2 if B > 4 else 0.0, seed=V % 89)
    s = synth.make_step(w, 0, DEV)
    if B > 4:
        s["gamma"][1], s["gamma"][B - 1] = 0, G + 1     # flagged rows, the last one among them
        s["temperature"][2] = float("nan")
        s["temperature"][3] = 0.0
    return w, s


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("B,G,V", [(1, 1, 4097), (2, 16, 4000), (5, 3, 4607), (16, 8, 8197), (33, 2, 65535), (148, 1, 12001), (255, 1, 9001),
                                   (256, 1, 8193), (257, 1, 8193), (3, 8, 128256)])
def test_direct_grids(dtype, B, G, V):
    w, s = _step(B, G, V, dtype)
    plan = plan_of(gpu_batch(s)._c(), "step")
    assert not plan["by_row"] and plan["direct"] == (B <= 256) and plan_of(gpu_batch(s)._c(), "signals")["direct"] == (B <= 256)
    assert plan["draw_ctas"] == {(1, "bf16"): 2, (2, "bf16"): 1, (33, "bf16"): 15, (33, "fp32"): 16, (3, "bf16"): 16, (148, "fp32"): 6}.get(
        (B, dtype), plan["draw_ctas"])
    gm, om = mlp_pair(synth.make_mlp(w, DEV))
    rows = np.arange(B) if B * G * V < 1 << 22 else np.unique(np.r_[0:min(B, 6), np.arange(0, B, max(1, B // 16)), B - 1])
    for _ in range(2):
        out = speckv.speckv_step(gpu_batch(s), s["comp"], gm)
    torch.cuda.synchronize()
    compare_step(out, oracle.step(oracle_batch(s, rows=rows), s["comp"].cpu().numpy()[rows], om), rows=rows)
    sig = speckv.speckv_signals(gpu_batch(s))
    for k in ("H", "C", "feat"):
        a, b = sig[k].cpu().numpy(), out[k].cpu().numpy()
        # cut into other ranges: sums of up to 2^17 fp32 terms in at least 256 chains
        assert np.allclose(a[sig["row_status"].cpu().numpy() == 0], b[sig["row_status"].cpu().numpy() == 0], rtol=1e-5, atol=1e-7), k


@pytest.mark.parametrize("B", [12, 100])
def test_waits_that_run_out(B):
    w, s = _step(B, 4, 20000, "bf16")
    s["uniforms"][:, :, 0] = 1.0 - 2.0 ** -24     # almost every walk ends in a rejection
    ref = {k: v.clone() for k, v in speckv.speckv_verify(gpu_batch(s)).items()}
    L = speckv.load_library()
    old = L.speckv_internal_set_wait_limit(1)     # one look at the record, which is not there yet
    try:
        out = {k: v.clone() for k, v in speckv.speckv_verify(gpu_batch(s)).items()}
        torch.cuda.synchronize()
    finally:
        L.speckv_internal_set_wait_limit(old)
    st, n = out["row_status"].cpu().numpy(), ref["n_accepted"].cpu().numpy()
    late = st == binding.ROW_TIMEOUT
    assert late.any() and (out["n_accepted"].cpu().numpy() == n).all()
    tok, want = out["out_tokens"].cpu().numpy(), ref["out_tokens"].cpu().numpy().copy()
    assert (ref["row_status"].cpu().numpy()[~late] == st[~late]).all()
    want[late, n[late]] = -1
    assert (tok == want).all()
    again = speckv.speckv_verify(gpu_batch(s))    # nothing of it stays
    assert all((again[k] == ref[k]).all() for k in ref)


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("B,G,V", [(24, 8, 9001), (98, 8, 20000), (256, 2, 8193), (256, 1, 20000), (40, 8, 65541)])
def test_next_gamma_over_this_steps_gamma(dtype, B, G, V):
    # grids of one to three rounds of CTAs: the later ones start when the first rows have already written their next gamma
    w, s = _step(B, G, V, dtype)
    gm, _ = mlp_pair(synth.make_mlp(w, DEV))
    bt = gpu_batch(s)
    assert plan_of(bt._c(), "step")["direct"] and not plan_of(bt._c(), "step_in_place")["direct"]
    apart = {k: v.clone() for k, v in speckv.speckv_step(bt, s["comp"], gm).items()}
    gamma = s["gamma"].clone()
    bt = gpu_batch(dict(s, gamma=gamma))
    out = speckv.StepOutputs.allocate(bt, gm.n_out)
    out.gamma_next = gamma
    for _ in range(4):
        gamma.copy_(s["gamma"])
        again = speckv.speckv_step(bt, s["comp"], gm, out=out)
        for k, v in apart.items():
            assert torch.equal(v.view(torch.int32), again[k].view(torch.int32)), k
