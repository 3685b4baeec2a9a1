"""Rows that start and end off the 16-byte grid: the sweep loads whole 16-byte granules and takes only a row's incomplete
first and last one element by element.  Vocabularies below one granule, of one granule, of whole and partial rounds of a
warp and of a CTA, rows cut into several slices whose last one is empty for some alignments, both types; the maximum, a
NaN and -inf placed in the edge elements.  Against the oracle under the rules of tests/parity.py."""
import numpy as np
import pytest
import torch

import oracle
import paper_2605_02888_b200 as speckv
from paper_2605_02888_b200 import synth

from parity import compare_step, gpu_batch, mlp_pair, oracle_batch

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _check(s, w):
    gm, om = mlp_pair(synth.make_mlp(w, DEV))
    out = speckv.speckv_step(gpu_batch(s), s["comp"], gm)
    torch.cuda.synchronize()
    compare_step(out, oracle.step(oracle_batch(s), s["comp"].cpu().numpy(), om))
    return out


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("V", [1, 3, 7, 9, 15, 17, 255, 257, 1023, 2047, 2049, 16385, 33333])
def test_rows_off_the_grid(dtype, V):
    w = synth.Workload("g", B=7, gamma_max=3, V=V, dtype=dtype, gamma_mode="ragged", temperature_mode="mixed",
                       sigma_d=(0.3, 0.6), seed=V)
    _check(synth.make_step(w, 0, DEV), w)


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("where", ["first", "last"])
def test_edge_elements_count(dtype, where):
    w = synth.Workload("g", B=6, gamma_max=2, V=5003, dtype=dtype, gamma_mode="fixed", gamma_fixed=2, temperature_mode="mixed",
                       sigma_d=(0.5,), seed=11)
    s = synth.make_step(w, 0, DEV)
    k = 0 if where == "first" else w.V - 1
    s["draft"][1:4, :, k] = 40.0     # the maximum sits in the row's edge granule
    s["target"][2:5, :, k] = 40.0
    s["draft_tokens"][1:4] = k
    s["target"][5, 0, k] = float("-inf")
    s["draft"][5, :, k] = float("-inf")
    _check(s, w)
    s["draft"][0, 1, k] = float("nan")
    s["target"][3, 0, k] = float("inf")
    out = _check(s, w)
    st = out["row_status"].cpu().numpy()
    assert np.array_equal(st, np.array([4, 0, 0, 4, 0, 0]))


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("jump", [30.0, 50.0, 300.0, 3.0e4])
def test_target_elements_far_above_the_reference(dtype, jump):
    # the sweep's reference is a maximum over its first loads; an element far above it, in one lane's later granules, makes
    # that lane's group sum large (30: below 2^60), beyond 2^60 (50) or infinite (300), and the group is read again
    w = synth.Workload("g", B=12, gamma_max=3, V=70001, dtype=dtype, gamma_mode="ragged", temperature=1.0, sigma_d=(0.5,), seed=5)
    s = synth.make_step(w, 0, DEV)
    for b in range(w.B):
        s["target"][b, :, 20000 + 4001 * b] = jump
        if b % 2:  # climbing: every group of the lane's raises the reference again
            s["target"][b, :, 30000:30000 + 60 * 512:512] += torch.arange(60, device=DEV).to(s["target"].dtype) * (jump / 60)
        if b % 3 == 0:
            s["draft"][b] = s["target"][b, :3]
            s["draft_tokens"][b] = 20000 + 4001 * b
    _check(s, w)


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 7, 8, 9, 17])
def test_draft_maxima_and_nans_in_every_step(dtype, n):
    # n steps per lane (pairs of them share a test for a new maximum): a maximum, a tie with it, or a NaN in each step of a lane
    step = 256 * 8 * n
    w = synth.Workload("g", B=2 * n + 1, gamma_max=3, V=step, dtype=dtype, gamma_mode="fixed", gamma_fixed=3, temperature=1.0,
                       sigma_d=(0.5,), seed=n)
    s = synth.make_step(w, 0, DEV)
    for b in range(2 * n):
        k = (b // 2) * 256 + 37 + b % 2
        s["draft"][b, 0, k] = 30.0
        s["draft"][b, 1, k] = 30.0
        s["draft"][b, 1, (k + 1) % step] = 30.0
        s["draft"][b, 1, (k + 300) % step] = 30.0
        s["draft"][b, 2, k: k + 700: 256] = 20.0 + torch.arange(s["draft"][b, 2, k: k + 700: 256].numel(), device=DEV).to(s["draft"].dtype)
    _check(s, w)
    s["draft"][0, 0, (n - 1) * 256 + 5] = float("nan")
    s["draft"][1, 2, (n // 2) * 256 + 5] = float("inf")
    st = _check(s, w)["row_status"].cpu().numpy()
    assert (st[:2] == 4).all() and (st[2:] == 0).all()
