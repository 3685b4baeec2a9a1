"""Short vocabularies, where one CTA takes a whole batch row: sizes around the limits of that choice, one to seventeen positions
(from eight warps per logit row to one, and more logit rows than warps), rows off the 16-byte grid, spans of one granule.
Against the oracle under the rules of tests/parity.py."""
import numpy as np
import pytest
import torch

import oracle
import paper_2605_02888_b200 as speckv
from paper_2605_02888_b200 import synth

from parity import compare_step, gpu_batch, mlp_pair, oracle_batch

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("B,G,V", [(9, 1, 4096), (9, 2, 4095), (40, 3, 4097), (5, 8, 4001), (255, 2, 8192), (256, 2, 8192),
                                   (256, 4, 8191), (256, 1, 8193), (300, 16, 2), (33, 16, 511), (1, 4, 1), (4, 16, 2979), (4, 16, 2978),
                                   (5, 16, 2979), (10, 16, 2305), (10, 16, 2304), (16, 16, 2816), (16, 16, 2817), (17, 16, 4096), (1024, 1, 15360),
                                   (1023, 1, 8193), (1024, 1, 15361), (2048, 1, 12289), (2048, 2, 15359), (2050, 2, 20480), (2050, 2, 20481)])
def test_step_and_its_parts(dtype, B, G, V):
    w = synth.Workload("s", B=B, gamma_max=G, V=V, dtype=dtype, gamma_mode="ragged", temperature_mode="mixed", sigma_t=1.0,
                       sigma_d=(0.2, 1.0, 2.0), frac_identical=0.2, seed=B + V)
    s = synth.make_step(w, 0, DEV)
    if B > 8:
        s["gamma"][1] = 0                       # flagged rows beside others
        s["temperature"][2] = -1.0
        s["target"][3, 0, V // 2] = float("nan")
        s["draft"][4, 0, V - 1] = float("inf")
        s["draft"][5, 0, : V - 1] = float("-inf")
    gm, om = mlp_pair(synth.make_mlp(w, DEV))
    batch = gpu_batch(s)
    out = {k: v.clone() for k, v in speckv.speckv_step(batch, s["comp"], gm).items()}
    torch.cuda.synchronize()
    compare_step(out, oracle.step(oracle_batch(s), s["comp"].cpu().numpy(), om))
    ver = speckv.speckv_verify(batch)
    for k in ("n_accepted", "out_tokens", "row_status"):
        assert torch.equal(ver[k], out[k]), k
    sig = speckv.speckv_signals(batch)
    ok = (out["row_status"] == 0).cpu().numpy()
    # the parts fold a row in other ranges: fp32 sums of up to V terms (tests/parity.py's tolerance)
    a, b = sig["feat"].cpu().numpy()[ok], out["feat"].cpu().numpy()[ok]
    assert (np.abs(a - b) <= 1e-5 * np.abs(b) + 1e-7).all()
