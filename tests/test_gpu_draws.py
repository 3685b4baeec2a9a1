"""The draws: a token located from span sums, the span narrowed down by a CTA.  Vocabularies for which a span is one granule
per lane, one level of 8 and of up to 64 parts and two levels deep; draft and target rows that sit differently on the 16-byte
grid; bonus draws (from the sweep's sums), residual draws, draws from p behind an empty residual, draft-side sampling.
Against the oracle under the rules of tests/parity.py, and against a cumulative sum in float64 where the oracle flags."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
import paper_2605_02888_b200 as speckv
from paper_2605_02888_b200 import synth, vocab_shard

from parity import compare_step, gpu_batch, mlp_pair, oracle_batch, plan_of

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


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("B,G,V", [(74, 8, 3000), (93, 8, 6001), (9, 8, 16380), (9, 8, 16384), (75, 8, 32767), (120, 5, 49151),
                                   (80, 8, 49153), (120, 5, 84032)])
def test_sampled_drafts_over_slices(dtype, B, G, V):
    # rows below and above 64 KB, as many as there are CTA slots and a few more; fp32 rows of one, two and three slices of 128 KB
    w = _workload(B, G, V, dtype)
    s = synth.make_step(w, 0, DEV)
    s["gamma"][:] = G
    u = torch.rand(B, G, device=DEV, generator=torch.Generator(DEV).manual_seed(V))
    rows = np.arange(0, B, max(1, B // 10))
    out = speckv.speckv_sample_draft(gpu_batch(s), u)
    ref = oracle.sample_draft(oracle_batch(s, rows=rows), u.cpu().numpy()[rows])
    clear = ref["near"] == 0
    # A uniform is flagged where it lies within 1e-6 of a boundary of the CDF: with a probability of at most the sum of
    # min(p, 2e-6) over the vocabulary, and a row with any of its G.  Rows are independent; four standard deviations and one row.
    p = torch.softmax(s["draft"][torch.as_tensor(rows, device=DEV)].double() / 0.9, -1)
    flagged = 1.0 - torch.prod(1.0 - p.clamp(max=2e-6).sum(-1), -1)
    most = float(flagged.sum() + 4.0 * (flagged * (1.0 - flagged)).sum().sqrt()) + 1.0
    assert (out["tokens"].cpu().numpy()[rows][clear] == ref["tokens"][clear]).all() and (~clear).sum() <= most
    assert (out["row_status"] == 0).all() and (out["tokens"] >= 0).all()


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("B,G,V", [(1, 1, 1), (1, 1, 255), (2, 3, 257), (1, 2, 2049), (1, 1, 32001), (1, 1, 65535), (2, 1, 65537),
                                   (1, 1, 200001), (300, 2, 1025), (100, 8, 33003), (40, 4, 151936), (200, 1, 300007)])
def test_sampling_stays_within_its_workspace(dtype, B, G, V):
    # exactly as many bytes as were asked for, what lies behind them unchanged: rows of fewer granules than a slice has lanes, the
    # most slices, unaligned rows, ranges in two to six pieces
    w = _workload(B, G, V, dtype)
    s = synth.make_step(w, 0, DEV)
    s["temperature"][::3] = 0.0
    u = torch.rand(B, G, device=DEV)
    batch = gpu_batch(s)
    n, c = ctypes.c_size_t(0), batch._c()
    assert (plan_of(c, "sample")["pieces"] > 1) == (B * V > 1000000)
    assert speckv.load_library().speckv_sample_workspace_size(ctypes.byref(c), ctypes.byref(n)) == 0
    mem = torch.full((n.value + 8192,), 0x5A, dtype=torch.uint8, device=DEV)
    a = speckv.speckv_sample_draft(batch, u, workspace=mem[:n.value])
    assert (mem[n.value:] == 0x5A).all()
    rows = np.arange(0, B, max(1, B // 20))
    ref = oracle.sample_draft(oracle_batch(s, rows=rows), u.cpu().numpy()[rows])
    clear = ref["near"] == 0
    assert (a["tokens"].cpu().numpy()[rows][clear] == ref["tokens"][clear]).all()


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


@pytest.mark.parametrize("B,G", [(1, 1), (256, 1), (911, 16), (3000, 16)])
def test_sampling_clears_its_counters(B, G):
    # fewer counters than one CTA clears, about a CTA's, just above and far above one pass of the clearing grid
    w = _workload(B, G, 40, "fp32")
    s = synth.make_step(w, 0, DEV)
    u = torch.rand(B, G, device=DEV)
    batch = gpu_batch(s)
    a = speckv.speckv_sample_draft(batch, u, workspace=torch.zeros(1 << 27, dtype=torch.uint8, device=DEV))
    b = speckv.speckv_sample_draft(batch, u, workspace=torch.full((1 << 27,), 0xFF, dtype=torch.uint8, device=DEV))
    assert torch.equal(a["tokens"], b["tokens"]) and torch.equal(a["row_status"], b["row_status"])
    assert ((b["tokens"] >= 0).sum(1) == s["gamma"]).all()


def test_calls_wait_for_their_inputs():
    # kernels that may be placed before their predecessor ends: inputs written right in front of each call, outputs read
    # right behind it, calls of different sizes one after the other without a synchronisation between them
    src = []
    for k, (B, G, V) in enumerate([(1, 4, 32000), (64, 4, 32000), (16, 8, 50257), (3, 2, 2000), (200, 4, 32001)]):
        w = _workload(B, G, V, "bf16" if k % 2 else "fp32")
        src.append([synth.make_step(w, i, DEV) for i in range(3)])
    gm, _ = mlp_pair(synth.make_mlp(w, DEV))

    def call(s):
        bt = gpu_batch(s)
        sig = speckv.speckv_signals(bt)
        got = [sig["feat"], speckv.speckv_select_gamma(sig["feat"], s["comp"], gm)["gamma_next"]]
        s["draft_tokens"].copy_(speckv.speckv_sample_draft(bt, s["uniforms"][:, :s["draft"].shape[1], 0].contiguous())["tokens"])
        r = speckv.speckv_step(bt, s["comp"], gm)
        return [x.clone() for x in got + [s["draft_tokens"], r["out_tokens"], r["n_accepted"], r["feat"], r["gamma_next"]]]

    def run(sync):
        bufs = [{k: v.clone() for k, v in x[0].items() if torch.is_tensor(v)} for x in src]
        outs = []
        for rep in range(12):
            for x, buf in zip(src, bufs):
                for k, v in buf.items():
                    v.copy_(x[rep % 3][k])
                if sync:
                    torch.cuda.synchronize()
                outs.append(call(dict(x[0], **buf)))
        torch.cuda.synchronize()
        return outs

    for a, b in zip(run(True), run(False)):
        for x, y in zip(a, b):
            assert torch.equal(x.nan_to_num(), y.nan_to_num())


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("B,V", [(1, 2000), (40, 4096), (300, 8000), (24, 9001)])
def test_calls_read_what_the_call_before_them_wrote(dtype, B, V):
    # gamma and the drafted tokens go from call to call in the buffers that the kernels wrote them to, with nothing launched
    # between (short vocabularies: the step is one kernel, the sampling kernel its direct predecessor; a vocabulary that is swept)
    w = synth.Workload("d", B=B, gamma_max=8, V=V, dtype=dtype, gamma_mode="choices", temperature=0.9, sigma_t=1.0,
                       sigma_d=(0.2, 1.0, 2.0), seed=V % 97)
    steps = [synth.make_step(w, i, DEV) for i in range(3)]
    gm, _ = mlp_pair(synth.make_mlp(w, DEV))

    def run(sync):
        done = torch.cuda.synchronize if sync else lambda: None
        gamma, tok = steps[0]["gamma"].clone(), torch.zeros_like(steps[0]["draft_tokens"])
        st = torch.empty(B, dtype=torch.int32, device=DEV)
        bts = [gpu_batch(dict(s, gamma=gamma, draft_tokens=tok)) for s in steps]
        us = [s["uniforms"][:, :8, 0].contiguous() for s in steps]
        outs = [speckv.StepOutputs.allocate(b, gm.n_out) for b in bts for _ in range(8)]
        for b, o in zip(bts * 8, outs):
            o.gamma_next = gamma  # the controller's choice is the next step's gamma
        toks = torch.zeros(len(outs), *tok.shape, dtype=torch.int32, device=DEV)
        ws = torch.empty(1 << 24, dtype=torch.uint8, device=DEV)
        done()
        for k, o in enumerate(outs):
            s, bt = steps[k % 3], bts[k % 3]
            speckv.speckv_sample_draft(bt, us[k % 3], tokens=tok, row_status=st, workspace=ws)
            done()
            speckv.speckv_step(bt, s["comp"], gm, out=o)
            done()
            toks[k].copy_(tok)
            f = speckv.speckv_signals(bt, out=o)["feat"]
            done()
            speckv.speckv_select_gamma(f, s["comp"], gm, scores=o.scores, gamma_next=gamma)
            done()
        torch.cuda.synchronize()
        assert all(int(o.row_status.abs().sum()) == 0 for o in outs)
        return [toks] + [t for o in outs for t in o.as_dict().values()]

    for a, b in zip(run(True), run(False)):
        assert torch.equal(a, b)


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("n,V", [(1, 3000), (2, 40001), (4, 40000)])
def test_shard_masses(dtype, n, V):
    # a rank's two masses at the stop position: of max(0, p - q) (0 where a bonus token is drawn) and of p
    B, G = 40, 2
    w = _workload(B, G, V, dtype, frac_identical=0.4)
    s = synth.make_step(w, 0, DEV)
    s["temperature"][::7] = 0.0
    full = gpu_batch(s)
    gm, _ = mlp_pair(synth.make_mlp(w, DEV))
    width, bounds = vocab_shard.shard_bounds(V, n)
    parts = [vocab_shard.slice_batch(full, a, e) for a, e in bounds]
    bufs = [vocab_shard.ShardBuffers.allocate(p, n, 4) for p in parts]
    for r, (p, o) in enumerate(zip(parts, bufs)):
        speckv.speckv_shard_sweep(p, bounds[r][0], o.state, o.tokl, o.workspace)
        bufs[0].all_state[r].copy_(o.state)
        bufs[0].all_tokl[r].copy_(o.tokl)
    o = bufs[0]
    speckv.speckv_shard_finish(parts[0], n, width, V, o.all_state, o.all_tokl, s["comp"], gm, o.out, o.row_info)
    stop = o.out.as_dict()["n_accepted"].long().cpu().numpy()
    for r, p in enumerate(parts):
        a, e = bounds[r]
        bufs[r].weight.fill_(7.0)
        speckv.speckv_shard_draw_sums(p, o.row_info, bufs[r].weight, bufs[r].workspace)
        got = bufs[r].weight.cpu().numpy()
        for b in range(B):
            T, k, g = float(s["temperature"][b]), int(stop[b]), int(s["gamma"][b])
            want = np.zeros(2)
            if T > 0:
                pt = torch.softmax(s["target"][b, k].double() / T, 0)
                want[1] = pt[a:e].sum()
                if k < g:
                    want[0] = (pt - torch.softmax(s["draft"][b, k].double() / T, 0)).clamp(min=0)[a:e].sum()
            # fp32 exponentials of fp32 arguments of up to ~30: 2e-6 of the mass of p, in differences too
            assert np.abs(got[b] - want).max() <= 5e-6 * max(want[1], 1e-3), (b, got[b], want)


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("B,G,V", [(100, 8, 16384), (100, 8, 16389), (100, 8, 33003), (100, 8, 65537), (95, 8, 70007), (40, 4, 151936)])
def test_sampled_drafts_from_pieces(dtype, B, G, V):
    # a warp's range in one, two and up to eight pieces; rows whose front is masked, and rows with elements at their end that lie more
    # than 2^60 above what the sums began with: the pieces summed before are brought to the new reference
    w = _workload(B, G, V, dtype)
    s = synth.make_step(w, 0, DEV)
    s["gamma"][:] = G
    s["draft"][::3, :, : V * 7 // 10] = float("-inf")
    s["draft"][1::3, :, V - 40:] += 60.0
    s["draft"][1::3, :, V * 9 // 16] += 59.0
    s["draft"][2::6, :, V - 1] += 100.0
    s["temperature"][5::7] = 0.0
    u = torch.rand(B, G, device=DEV, generator=torch.Generator(DEV).manual_seed(V))
    u[:, 0], u[:, 1] = 0.0, 1.0 - 2.0 ** -24
    rows = np.arange(0, B, 11)
    out = speckv.speckv_sample_draft(gpu_batch(s), u)
    ref = oracle.sample_draft(oracle_batch(s, rows=rows), u.cpu().numpy()[rows])
    tok, want = out["tokens"].cpu().numpy()[rows], ref["tokens"]
    # The oracle flags a row where any of its uniforms is near a boundary, as the two imposed ones are; here each position by itself,
    # from a cumulative sum in 64 bits.  A uniform is near one with a probability of at most sum(min(p, 2e-6)).
    at = torch.as_tensor(rows, device=DEV)
    p = torch.softmax(s["draft"][at].double() / 0.9, -1)
    cdf = p.cumsum(-1)
    x = u[at].double().unsqueeze(-1) * cdf[..., -1:]
    greedy = (s["temperature"].cpu().numpy()[rows] == 0.0)[:, None]
    clear = ((cdf - x).abs().amin(-1) > 1e-6).cpu().numpy() | greedy
    assert (tok[clear] == want[clear]).all()
    # the two imposed uniforms: a token that may be drawn, with nothing to speak of in front of it and behind it respectively
    got = torch.as_tensor(tok, device=DEV)[:, :2].long().unsqueeze(-1)
    share, upto = p[:, :2].gather(-1, got).squeeze(-1), (cdf[:, :2] / cdf[:, :2, -1:]).gather(-1, got).squeeze(-1)
    sampled = torch.as_tensor(~greedy[:, 0], device=DEV)
    assert (share[sampled] > 0).all() and (upto - share)[sampled, 0].max() <= 1e-6 and (1.0 - upto)[sampled, 1].max() <= 1e-6
    near = p.clamp(max=2e-6).sum(-1)[:, 2:]
    assert (~clear[:, 2:]).sum() <= float(near.sum() + 4.0 * near.sum().sqrt()) + 1.0
    assert (out["row_status"] == 0).all() and (out["tokens"] >= 0).all()
