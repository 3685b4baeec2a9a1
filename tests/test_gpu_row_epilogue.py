"""The row epilogue of the sweep: positions shared out over the eight warps of a CTA, a logit row's partials over half a warp
(two per lane beyond 16).  Batches whose rows are cut into 1, 2, 9, 15, 16, 17, 31 and 32 slices (asserted) and whose positions
fill the eight warps once, exactly and more than twice, greedy and sampled rows, against the oracle under the rules of
tests/parity.py."""
import pytest
import torch

import oracle
import paper_2605_02888_b200 as speckv
from paper_2605_02888_b200 import synth

from parity import compare_step, gpu_batch, mlp_pair, oracle_batch, plan_of

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("slices,B,G", [(1, 40, 16), (2, 21, 12), (9, 2, 12), (15, 1, 9), (15, 2, 4), (16, 1, 16), (16, 2, 8), (17, 1, 16),
                                        (17, 3, 3), (31, 1, 8), (32, 1, 8), (32, 1, 1), (32, 2, 3)])
def test_epilogue_over_slices_and_positions(dtype, slices, B, G):
    # a slice of one granule per lane, or of five where a row has too few of them for the batch to be cut
    V = slices * 256 * (8 if dtype == "bf16" else 4) * (5 if slices <= 2 else 1)
    w = synth.Workload("e", B=B, gamma_max=G, V=V, dtype=dtype, gamma_mode="fixed", gamma_fixed=G, temperature_mode="mixed",
                       sigma_d=(0.3, 0.6), frac_onehot=0.2, frac_identical=0.3, seed=B + G)
    for step in range(2):
        s = synth.make_step(w, step, DEV)
        plan = plan_of(gpu_batch(s)._c(), "step")
        assert not plan["by_row"] and plan["slices"] == slices, plan
        gm, om = mlp_pair(synth.make_mlp(w, DEV))
        out = speckv.speckv_step(gpu_batch(s), s["comp"], gm)
        torch.cuda.synchronize()
        compare_step(out, oracle.step(oracle_batch(s), s["comp"].cpu().numpy(), om))


# sizes whose slices and positions do not come out even, rows off the 16-byte grid among them
@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("B,G,V", [(40, 16, 1000), (5, 8, 40000), (9, 4, 40000), (5, 7, 40000), (4, 8, 40001), (1, 1, 66000),
                                   (2, 16, 66000), (1, 9, 66000)])
def test_epilogue_over_uneven_sizes(dtype, B, G, V):
    w = synth.Workload("e", B=B, gamma_max=G, V=V, dtype=dtype, gamma_mode="fixed", gamma_fixed=G, temperature_mode="mixed",
                       sigma_d=(0.3, 0.6), frac_onehot=0.2, frac_identical=0.3, seed=B + G)
    for step in range(2):
        s = synth.make_step(w, step, DEV)
        gm, om = mlp_pair(synth.make_mlp(w, DEV))
        out = speckv.speckv_step(gpu_batch(s), s["comp"], gm)
        torch.cuda.synchronize()
        compare_step(out, oracle.step(oracle_batch(s), s["comp"].cpu().numpy(), om))
