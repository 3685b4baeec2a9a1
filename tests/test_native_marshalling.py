"""The native argument marshalling: it refuses (and leaves to the Python path, which raises) whatever the Python checks
refuse, and makes the same call for everything else."""
import dataclasses
import os

import pytest
import torch

import paper_2605_02888_b200 as speckv
from paper_2605_02888_b200 import binding, build, synth

from parity import gpu_batch, mlp_pair

DEV = "cuda:0"


def _native():
    nat, addr = binding._entry(speckv.load_library())
    assert nat, "the native marshalling module could not be built or loaded"
    return nat, addr


def test_cpu_tensors_and_odd_objects_are_left_to_the_python_path():
    nat, addr = _native()
    b = speckv.Batch(draft_logits=torch.zeros(2, 2, 8), target_logits=torch.zeros(2, 3, 8))
    for bad in (b, dataclasses.replace(b, draft_logits=None), object(), None):
        assert nat.verify(addr["speckv_verify"], addr["speckv_workspace_size"], bad, object()) is None
        assert nat.sample(addr["speckv_sample_draft"], addr["speckv_sample_workspace_size"], bad, None, None, None, None) is None
    with pytest.raises(TypeError):
        nat.step(addr["speckv_step"])
    with pytest.raises(ValueError):
        speckv.speckv_sample_draft(b, torch.zeros(2, 2))


def test_a_module_built_for_another_torch_is_not_loaded(monkeypatch):
    here = build.torch_lib_path()
    for name, value in (("__version__", "9.9.9+cu999"), ("compiled_with_cxx11_abi", lambda abi=torch.compiled_with_cxx11_abi(): not abi)):
        with monkeypatch.context() as m:
            m.setattr(torch, name, value)
            other = build.torch_lib_path()
            assert other != here and not os.path.exists(other)
            # it would have to be built; where that fails the Python path does the calls
            m.setattr(build.subprocess, "check_call", lambda *a, **k: (_ for _ in ()).throw(OSError("no compiler")))
            m.setattr(binding, "_native", None)
            with pytest.warns(UserWarning, match="native argument marshalling"):
                assert binding._entry(speckv.load_library())[0] is False
    assert build.torch_lib_path() == here


@pytest.mark.gpu
def test_what_the_python_checks_refuse_is_refused():
    nat, addr = _native()
    w = synth.Workload("t", B=6, gamma_max=3, V=1000, dtype="bf16", gamma_mode="ragged", temperature=0.9, seed=2)
    s = synth.make_step(w, 0, DEV)
    gm, _ = mlp_pair(synth.make_mlp(w, DEV))
    bt = gpu_batch(s)
    out = speckv.StepOutputs.allocate(bt, 4)
    go = lambda b=bt, c=s["comp"], m=gm, o=out: nat.step(addr["speckv_step"], addr["speckv_workspace_size"], b, c, m, o)
    assert go() == binding.OK
    r = dataclasses.replace
    for b in (r(bt, gamma=s["gamma"].long()), r(bt, gamma=s["gamma"][:5]), r(bt, temperature=s["temperature"].double()),
              r(bt, uniforms=s["uniforms"][:, :3]), r(bt, target_logits=s["target"][:, :3]), r(bt, target_logits=s["target"].float()),
              r(bt, draft_logits=s["draft"].half()), r(bt, draft_tokens=s["draft_tokens"].t().contiguous().t()),
              r(bt, draft_logits=s["draft"].transpose(1, 2)), r(bt, uniforms=s["uniforms"].cpu())):
        assert go(b=b) is None
        with pytest.raises((ValueError, TypeError)):
            speckv.speckv_step(b, s["comp"], gm, out=out)
    for o in (r(out, H=out.H[:, :2]), r(out, n_accepted=out.n_accepted.float()), r(out, workspace=out.workspace[:256]),
              r(out, out_tokens=out.out_tokens.cpu()), r(out, scores=out.scores[:, :3])):
        assert go(o=o) is None
        with pytest.raises((ValueError, TypeError)):
            speckv.speckv_step(bt, s["comp"], gm, out=o)
    for m in (r(gm, b1=gm.b1[:3]), r(gm, W2=gm.W2.double()), r(gm, gamma_choices=(2, 4))):
        assert go(m=m) is None
        with pytest.raises((ValueError, TypeError)):
            speckv.speckv_step(bt, s["comp"], m, out=out)
    assert go(c=s["comp"][:, :1]) is None


@pytest.mark.gpu
def test_native_and_python_calls_agree(monkeypatch):
    w = synth.Workload("t", B=9, gamma_max=4, V=3001, dtype="fp32", gamma_mode="ragged", temperature_mode="mixed", seed=3)
    s = synth.make_step(w, 0, DEV)
    gm, _ = mlp_pair(synth.make_mlp(w, DEV))
    u = torch.rand(w.B, w.gamma_max, device=DEV)

    def calls():
        out = speckv.speckv_step(gpu_batch(s, entropy_in_bits=True), s["comp"], gm)
        sig = speckv.speckv_signals(gpu_batch(s, temperature_scalar=0.7))
        ctl = speckv.speckv_select_gamma(sig["feat"], s["comp"], gm)
        ver = speckv.speckv_verify(gpu_batch(s, flags=binding.READ_ALL_TARGET_ROWS))
        smp = speckv.speckv_sample_draft(gpu_batch(s), u)
        torch.cuda.synchronize()
        return [t.clone() for d in (out, sig, ctl, ver, smp) for t in d.values()]
    a = calls()
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):   # the current stream is the one that is used
        b = calls()
    monkeypatch.setattr(binding, "_native", False)
    c = calls()
    for x, y, z in zip(a, b, c):
        assert torch.equal(x, y) and torch.equal(x, z)
