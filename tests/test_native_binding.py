"""The calling thread's part in C++ (csrc/sd_native.cpp): what it takes it answers as the general way does, and it
leaves everything else to that way."""
import os
import subprocess
import sys
import types

import pytest
import torch

from paper_2603_12617_b200 import binding, shard

NONE = types.SimpleNamespace(**{n: (lambda *a: None) for n in ("step", "hint", "greedy", "errors", "ensemble", "lmhead", "vp_partial",
                                                               "vp_finish", "vp_draw")})


def test_anything_but_device_tensors_is_left_to_the_general_way():
    T, D = torch.zeros(1, 3, 8), torch.zeros(1, 2, 8)
    x, u = torch.zeros(1, 2, dtype=torch.int32), torch.zeros(1, 3)
    n = binding._native
    assert n.step(T, D, x, u, 1.0, True, True) is None
    assert n.step(T, D, x, u, 1.0) is None and n.step(None, 1, "x", [], {}, True, True) is None
    assert n.greedy(T, x, True) is None and n.errors(T, D, x, u, 1.0, True, True, True) is None
    assert n.hint(T, D, x, u, 1.0, D, T) is None and n.ensemble(T, [D], 1.0, 1.0, None, True, False) is None
    assert n.lmhead(D[0], D[0]) is None and n.vp_partial(T, D, x, 1.0, 0, 8, T, None) is None
    assert n.vp_finish(T, D, x, u, 1.0, 0, 8, T, 1, 0, T, True, True) is None
    assert n.vp_draw(T, D, x, u, 1.0, 0, 8, x, T, 1, 0, x, T) is None
    with pytest.raises(ValueError):
        binding.sd_verify_feedback(T, D, x, u, 1.0)
    with pytest.raises(TypeError):
        n.bind(1, 2)


def test_a_build_against_another_torch_is_not_loaded(monkeypatch):
    monkeypatch.setattr(torch, "__version__", "0.0.1")
    with pytest.raises(ImportError, match="0.0.1"):
        binding._load_native()


def test_the_build_makes_one_for_the_torch_that_runs(monkeypatch):
    import __graft_entry__ as entry
    entry.build()
    ran = []
    monkeypatch.setattr(entry.subprocess, "Popen", lambda c: types.SimpleNamespace(wait=lambda: ran.append(c) or 0, returncode=0))
    entry.build()
    assert ran == []                                             # everything is there
    monkeypatch.setattr(torch, "__version__", "0.0.1")
    entry.build()
    assert len(ran) == 1 and ran[0][0] == "g++" and "0.0.1" in ran[0][ran[0].index("-o") + 1]


def flat(o):
    if isinstance(o, torch.Tensor) or o is None:
        return [o]
    if isinstance(o, (list, tuple)):
        return [t for v in o for t in flat(v)]
    return [t for v in vars(o).values() for t in flat(v)]


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_same_answers_as_the_general_way(dtype, monkeypatch):
    B, k, V = 3, 2, 4096
    g = torch.Generator(device="cuda").manual_seed(3)
    T = torch.randn(B, k + 1, V, device="cuda", generator=g).to(dtype)
    D = torch.randn(B, k, V, device="cuda", generator=g).to(dtype)
    x = torch.randint(0, V, (B, k), device="cuda", dtype=torch.int32, generator=g)
    u = torch.rand(B, k + 1, device="cuda", generator=g)
    code = binding._dtype_code(T)
    cum = torch.rand(2, device="cuda", dtype=torch.float64, generator=g)
    ws = torch.empty(binding.sd_hint_workspace_bytes(B, k, V, code), dtype=torch.uint8, device="cuda")
    vws = torch.empty(binding.sd_vp_workspace_bytes(B, k, V, code), dtype=torch.uint8, device="cuda")
    calls = {
        "step": lambda T=T, x=x, tau=0.8: binding.sd_verify_feedback(T, D, x, u, tau),
        "step without": lambda: binding.sd_verify_feedback(T, D, x, u, 1, want_loss=False, want_grad=False),
        "greedy": lambda T=T: binding.sd_verify_greedy(T, x),
        "greedy without": lambda: binding.sd_verify_greedy(T, x, want_argmax=False),
        "errors": lambda: binding.sd_verify_error_feedback(T, D, x, u, 0.8),
        "errors without": lambda: binding.sd_verify_error_feedback(T, D, x, u, 0.8, want_loss=False, want_grad=False, want_status=False),
        "hint": lambda: binding.sd_verify_feedback_hint(T, D, x, u, 0.8, D, workspace=ws),
        "ensemble": lambda: binding.sd_ensemble_feedback(T, [D, D], 0.8, 10.0, cum_loss=cum, want_status=True),
        "ensemble without": lambda: binding.sd_ensemble_feedback(T, (D,), 0.8, 10, want_grad=False),
        "lmhead": lambda: binding.sd_lmhead_grad(D.bfloat16().view(B * k, V), T[0, :1, :64].bfloat16().expand(B * k, 64).contiguous()),
    }

    def vp():
        rec = binding.sd_vp_partial(T, D, x, 0.8, 0, V, vws)
        f = binding.sd_vp_finish(T, D, x, u, 0.8, 0, V, rec, 1, 0, vws)
        return rec, f, binding.sd_vp_draw(T, D, x, u, 0.8, 0, V, f.accept_len, f.local_mass, 1, 0, f.status, vws)
    calls["vp"] = vp
    native = binding._native
    for name, call in calls.items():
        with monkeypatch.context() as m:
            m.setattr(binding, "_native", NONE)
            want = flat(call())
        got = flat(call())
        torch.cuda.synchronize()
        assert len(got) == len(want), name
        for a, b in zip(got, want):
            assert (a is None) == (b is None), name
            if a is not None:
                assert (a.dtype, a.shape, a.stride(), a.device) == (b.dtype, b.shape, b.stride(), b.device), name
                assert torch.equal(a.contiguous().view(torch.uint8), b.contiguous().view(torch.uint8)), name
    # taken only as they are: no views of other layouts, no subclasses, nothing that raises the general way
    class Mine(torch.Tensor):
        pass
    assert native.step(T, D, x, u, 0.8, True, True) is not None
    for bad in ((T.transpose(0, 1).contiguous().transpose(0, 1), x), (T, x.long()), (T.as_subclass(Mine), x), (T[:, :2], x)):
        assert native.step(bad[0], D, bad[1], u, 0.8, True, True) is None
        assert native.greedy(bad[0], bad[1], True) is None or bad[0].shape[1] == 2
    assert native.step(T, D, x, u, "1", True, True) is None
    with pytest.raises(ValueError):
        binding.sd_verify_feedback(T, D, x.long(), u, 0.8)
    with pytest.raises(binding.SdVerifyError):
        binding.sd_verify_feedback(T, D, x, u, 0.0)
    assert shard.vocab_cuts(V, 1, T.element_size())[0] == (0, V)


@pytest.mark.gpu
@pytest.mark.parametrize("way", ["C++", "general"])
def test_buffers_of_the_vocabulary_parallel_step_that_are_too_small_or_of_another_type(way, monkeypatch):
    """What the kernels would read or write from a tensor's first entry on has to be there; more room is fine."""
    B, k, V = 3, 2, 4096
    g = torch.Generator(device="cuda").manual_seed(5)
    T, D = torch.randn(B, k + 1, V, device="cuda", generator=g), torch.randn(B, k, V, device="cuda", generator=g)
    x = torch.randint(0, V, (B, k), device="cuda", dtype=torch.int32, generator=g)
    u = torch.rand(B, k + 1, device="cuda", generator=g)
    ws = torch.empty(binding.sd_vp_workspace_bytes(B, k, V, binding.SD_DTYPE_F32), dtype=torch.uint8, device="cuda")
    if way == "general":
        monkeypatch.setattr(binding, "_native", NONE)
    rows = B * (k + 1)
    records = binding.sd_vp_partial(T, D, x, 0.8, 0, V, ws)
    room = torch.full((rows + 2, 48), 7, dtype=torch.uint8, device="cuda")
    assert binding.sd_vp_partial(T, D, x, 0.8, 0, V, ws, out_records=room) is room
    assert torch.equal(room[:rows], records) and (room[rows:] == 7).all()
    for bad in (records[:-1], torch.empty(rows, 96, dtype=torch.uint8, device="cuda")[:, :48], torch.empty(0, dtype=torch.uint8, device="cuda")):
        with pytest.raises(ValueError):
            binding.sd_vp_partial(T, D, x, 0.8, 0, V, ws, out_records=bad)
    with pytest.raises(ValueError):
        binding.sd_vp_partial(T, D, x.long(), 0.8, 0, V, ws)
    f = binding.sd_vp_finish(T, D, x, u, 0.8, 0, V, records, 1, 0, ws)
    for bad in (u.double(), u[:, :k].contiguous(), u.t()):
        with pytest.raises(ValueError):
            binding.sd_vp_finish(T, D, x, bad, 0.8, 0, V, records, 1, 0, ws)
        with pytest.raises(ValueError):
            binding.sd_vp_draw(T, D, x, bad, 0.8, 0, V, f.accept_len, f.local_mass, 1, 0, f.status, ws)
    with pytest.raises(ValueError):
        binding.sd_vp_finish(T, D, x, u, 0.8, 0, V, records.expand(1, rows, 48)[:, :1].expand(1, rows, 48), 1, 0, ws)
    n, st = f.accept_len, f.status
    want = binding.sd_vp_draw(T, D, x, u, 0.8, 0, V, n, f.local_mass, 1, 0, st, ws)
    for good in ((n, None), (n, st.view(torch.uint32)), (torch.cat([n, n]), torch.cat([st, st]))):
        assert torch.equal(binding.sd_vp_draw(T, D, x, u, 0.8, 0, V, good[0], f.local_mass, 1, 0, good[1], ws), want)
    for bad in ((n.long(), st), (n[:-1], st), (n.float(), st), (n, st.long()), (n, st[:-1]), (n, st.float())):
        with pytest.raises(ValueError):
            binding.sd_vp_draw(T, D, x, u, 0.8, 0, V, bad[0], f.local_mass, 1, 0, bad[1], ws)
    with pytest.raises(ValueError):
        binding.sd_vp_draw(T, D, x, u, 0.8, 0, V, n, f.local_mass[:1].expand(B, 2), 1, 0, st, ws)
    torch.cuda.synchronize()


# A process of its own: an exception that gets out without the interpreter's lock takes the interpreter with it.
REFUSING = """
import threading, torch
from paper_2603_12617_b200 import binding as b
T, D = torch.zeros(2, 3, 4096, device="cuda"), torch.zeros(2, 2, 4096, device="cuda")
x, u = torch.zeros(2, 2, dtype=torch.int32, device="cuda"), torch.zeros(2, 3, device="cuda")
G, X = torch.zeros(4, 64, dtype=torch.bfloat16, device="cuda"), torch.zeros(4, 64, dtype=torch.bfloat16, device="cuda")
ws = torch.empty(1 << 20, dtype=torch.uint8, device="cuda")
rec = b.sd_vp_partial(T, D, x, 1.0, 0, 4096, ws)
f = b.sd_vp_finish(T, D, x, u, 1.0, 0, 4096, rec, 1, 0, ws)
bad = lambda t: (torch._C._set_throw_on_mutable_data_ptr(t), t)[1]
calls = [lambda v: b.sd_verify_feedback(T, D, x, v, 1.0), lambda v: b.sd_verify_feedback(T.bfloat16(), D.bfloat16(), x, v, 1.0),
         lambda v: b.sd_verify_feedback_hint(T, D, x, v, 1.0, D, workspace=ws), lambda v: b.sd_verify_error_feedback(T, D, x, v, 1.0),
         lambda v: b.sd_vp_finish(T, D, x, v, 1.0, 0, 4096, rec, 1, 0, ws),
         lambda v: b.sd_vp_draw(T, D, x, v, 1.0, 0, 4096, f.accept_len, f.local_mass, 1, 0, f.status, ws)]
with_x = [lambda v: b.sd_verify_greedy(T, v), lambda v: b.sd_vp_partial(T, D, v, 1.0, 0, 4096, ws)]
with_D = [lambda v: b.sd_ensemble_feedback(T, [D, v], 1.0, 10.0)]
with_X = [lambda v: b.sd_lmhead_grad(G, v)]
done = 0
for group, t in ((calls, u), (with_x, x), (with_D, D), (with_X, X)):
    for call in group:
        call(t)
        try:
            call(bad(t.clone()))
        except RuntimeError as e:
            assert "data pointer" in str(e), e
            done += 1
        ran = []
        th = threading.Thread(target=lambda: ran.append(1))      # the lock is where it belongs
        th.start()
        th.join()
        assert ran
        call(t)
torch.cuda.synchronize()
print("refused", done)
"""


@pytest.mark.gpu
def test_tensors_that_refuse_their_address_raise():
    """The address of a tensor is asked for while the interpreter's lock is held: a refusal is an exception like any other."""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    env = dict(os.environ, PYTHONPATH=os.pathsep.join([root, os.environ.get("PYTHONPATH", "")]))
    r = subprocess.run([sys.executable, "-c", REFUSING], env=env, cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "refused 10" in r.stdout, r.stdout + r.stderr
