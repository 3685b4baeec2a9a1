"""The row epilogue of the sliced sweep: positions shared out over the eight warps of a CTA, a logit row's partials
over half a warp (two per lane beyond 16).  Batches whose rows are cut into 1, 14, 15, 16, 18 and 32 slices and whose
positions fill the eight warps once, exactly and more than twice, greedy and sampled rows, against the oracle under
the rules of tests/parity.py."""
import pytest
import torch

import oracle
import paper_2605_02888_b200 as speckv
from paper_2605_02888_b200 import synth

from parity import compare_step, gpu_batch, mlp_pair, oracle_batch

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


# slices per logit row = min(32, ceil(1184 / (B * (2G+1))), V / 2048) for these sizes
@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("B,G,V", [(40, 16, 1000), (5, 8, 40000), (9, 4, 40000), (5, 7, 40000), (4, 8, 40001), (1, 1, 66000),
                                   (2, 16, 66000), (1, 9, 66000)])
def test_epilogue_over_slices_and_positions(dtype, B, G, V):
    w = synth.Workload("e", B=B, gamma_max=G, V=V, dtype=dtype, gamma_mode="fixed", gamma_fixed=G, temperature_mode="mixed",
                       sigma_d=(0.3, 0.6), frac_onehot=0.2, frac_identical=0.3, seed=B + G)
    for step in range(2):
        s = synth.make_step(w, step, DEV)
        gm, om = mlp_pair(synth.make_mlp(w, DEV))
        out = speckv.speckv_step(gpu_batch(s), s["comp"], gm)
        torch.cuda.synchronize()
        compare_step(out, oracle.step(oracle_batch(s), s["comp"].cpu().numpy(), om))
