"""How a call is cut into CTAs and warps, over sizes, types and alignments: every granule of a row belongs to a warp, whatever
the rule gives, and the partials, span sums and draw sums fit the places that the workspace has for them.  Host arithmetic, no GPU."""
import ctypes as C
import random

import pytest

import paper_2605_02888_b200 as speckv
from paper_2605_02888_b200 import binding

from parity import plan_of


def batch(B, G, V, dtype, offset=0, pad=0):
    """offset: elements by which the logits start off a 16-byte boundary; pad: elements between rows"""
    b = binding._CBatch()
    es = 2 if dtype == "bf16" else 4
    b.B, b.gamma_max, b.V, b.dtype = B, G, V, binding.BF16 if dtype == "bf16" else binding.F32
    b.draft_logits = b.target_logits = 0x10000 + offset * es
    b.draft_stride_pos = b.target_stride_pos = V + pad
    b.draft_stride_b, b.target_stride_b = G * (V + pad), (G + 1) * (V + pad)
    b.draft_tokens = b.uniforms = 0x10000
    b.temperature_scalar = 1.0
    return b


def check(b, call):
    p = plan_of(b, call)
    E = 8 if b.dtype == binding.BF16 else 4
    aligned = all(x % 16 == 0 for x in (b.draft_logits, b.draft_stride_pos * 16 // E, b.draft_stride_b * 16 // E)) and \
        (call != "step" or (b.target_stride_b * 16 // E) % 16 == 0)
    ng = -(-b.V // E) if aligned else (b.V + 2 * (E - 1)) // E   # granules a row can touch
    warps = p["slices"] if p["by_row"] else 8 * p["slices"]
    assert warps * p["per_warp"] >= ng, (p, ng)
    assert 1 <= p["slices"] <= 32 and p["spans"] <= warps * p["pieces"]
    assert p["pieces"] * p["piece"] >= p["per_warp"]     # every granule of a range is in one of its pieces
    if p["by_row"]:
        assert call != "sample" and 8 % p["slices"] == 0 and p["spans"] == p["slices"]
    else:
        assert p["per_warp"] >= 32 and p["per_warp"] % 32 == 0
        assert p["spans"] // p["pieces"] * p["per_warp"] >= ng   # a warp without a place for its sum has no granule
    if call == "step":
        # 16 bytes for each of a direct grid's sums, 8 for another's, in 32 * 8 places of 8
        assert 1 <= p["draw_ctas"] <= (16 if p["direct"] else 32) and p["draw_ctas"] * 8 * p["draw_per_warp"] >= ng
        # arrivals of a position: the slices of two rows; places for all tests in a word of 64 bits
        assert p["tests"] == 0 or (2 * p["slices"] < 1 << p["pos_bits"] and p["tests"] * p["pos_bits"] <= 64)
        assert not (p["direct"] and (p["by_row"] or p["tests"] or b.B > 256))
    else:
        assert p["tests"] == 0 and p["pieces"] <= (8 if call == "sample" else 1)
    if call == "sample":
        assert p["spans"] <= 256 and not p["direct"] and (p["pieces"] == 1 or p["spans"] % p["pieces"] == 0)
        n = C.c_size_t(0)
        assert speckv.load_library().speckv_sample_workspace_size(C.byref(b), C.byref(n)) == 0
        assert n.value >= 4 * (b.B * b.gamma_max + 2 * b.B) + 8 * b.B * b.gamma_max * p["spans"]
    return p


@pytest.mark.parametrize("call", ["signals", "step", "sample"])
def test_every_granule_has_a_warp(call):
    rnd = random.Random(5)
    edges = [1, 7, 8, 9, 255, 256, 257, 4095, 4096, 4097, 8191, 8192, 8193, 12288, 12289, 15360, 15361, 16383, 20480, 20481, 32000, 32768,
             50257, 128256, 151936, 1 << 20, (1 << 24) + 5]
    seen, how = set(), set()
    for k in range(4000):
        V = rnd.choice(edges) if k % 2 else int(2 ** rnd.uniform(0, 21))
        B, G = int(2 ** rnd.uniform(0, 12)), rnd.randint(1, 16)
        dtype = rnd.choice(["bf16", "fp32"])
        p = check(batch(B, G, V, dtype, offset=rnd.choice([0, 0, 1, 3]), pad=rnd.choice([0, 0, 8, 5])), call)
        seen.add(("row", p["slices"]) if p["by_row"] else p["slices"])
        how.add((p["direct"], p["tests"], p["pos_bits"], p["rows_major"]) if call == "step" and not p["by_row"] else p["pieces"])
    assert {1, 2, 15, 16, 17, 32} <= seen and {("row", n) for n in {"signals": (1, 2, 4, 8), "step": (1, 2)}.get(call, ())} <= seen, seen
    if call == "step":   # direct; a list without tests; of two positions by row and by position; of all, with counters of 4 and 8 bits
        assert {(1, 0, 0, 0), (0, 0, 0, 0), (0, 2, 4, 1), (0, 2, 4, 0), (0, 16, 4, 0), (0, 8, 8, 0)} <= how, how
    if call == "sample":
        assert {1, 2, 3, 5, 8} <= how, how


def test_which_batches_take_a_cta_per_row():
    by_row = lambda call, B, G, V: bool(plan_of(batch(B, G, V, "fp32"), call)["by_row"])
    # short rows in small batches; few of them with many positions go through the sweep
    assert by_row("step", 1, 8, 4096) and not by_row("step", 1, 8, 4097)
    assert not by_row("step", 4, 16, 4000) and by_row("step", 4, 16, 2978) and by_row("step", 5, 16, 4000)
    assert not by_row("signals", 4, 12, 4000) and by_row("signals", 4, 8, 4000) and by_row("signals", 40, 16, 4096)
    # longer ones with more rows
    assert by_row("step", 256, 8, 8192) and not by_row("step", 255, 8, 8192)
    assert by_row("step", 1024, 8, 15360) and not by_row("step", 1024, 8, 15361) and not by_row("step", 4096, 8, 15361)
    assert by_row("signals", 2048, 2, 20480) and not by_row("signals", 2048, 1, 20480)
    assert not any(plan_of(batch(B, 4, V, "bf16"), "sample")["by_row"] for B in (1, 64, 4096) for V in (100, 4000, 9000))


def test_a_step_that_writes_over_its_gamma_takes_a_list():
    # CTAs that find their work from the gamma of all rows would see what the first rows' epilogues have written
    for B, G, V, dtype in [(1, 4, 32000, "fp32"), (100, 8, 20000, "bf16"), (98, 8, 20000, "fp32"), (256, 1, 8193, "bf16"), (37, 8, 50257, "bf16")]:
        b = batch(B, G, V, dtype)
        b.gamma = 0x20000
        b.temperature = 0x30000
        assert plan_of(b, "step")["direct"] and plan_of(b, "signals")["direct"]
        in_place = plan_of(b, "step_in_place")
        assert not in_place["direct"] and not in_place["by_row"]
        assert {k: in_place[k] for k in ("slices", "per_warp", "spans")} == {k: plan_of(b, "step")[k] for k in ("slices", "per_warp", "spans")}
    assert plan_of(batch(100, 8, 20000, "bf16"), "step_in_place")["direct"]   # gamma_max for all rows: nothing to write over
