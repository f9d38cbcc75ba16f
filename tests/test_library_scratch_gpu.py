"""The library's own scratch (calls without a workspace) under CUDA graphs and after a wait that ran out:
what the host believes of its contents must hold whenever a call runs, not only when it was issued.
Every answer is compared, bit for bit, with the call on a fresh caller workspace."""
import ctypes
import types

import pytest
import torch

from paper_2603_12617_b200 import synth
from test_parity_gpu import to_device

pytestmark = pytest.mark.gpu


@pytest.fixture()
def binding():
    import __graft_entry__ as entry
    entry.build()
    from paper_2603_12617_b200 import binding as b
    b.sd_release_cached_buffers()
    yield b
    b.sd_release_cached_buffers()


LARGE = (64, 4, 32768, "bf16")       # the two sweeps; counters where SMALL keeps accept flags and row constants
SMALL = (8, 3, 8192, "f32")          # the cluster kernel, in the same scratch


class Call:
    """One call on the library's scratch with output tensors of its own, and the answer it must give."""

    def __init__(self, binding, kind, shape, index):
        B, k, V, dtype = shape
        inp = synth.make_inputs(synth.custom_config(B=B, k=k, V=V, dtype=dtype, tau=0.9, index=index))
        self.args = T, D, x, u = to_device(inp)
        tau = inp.tau
        if kind == "step":
            want = binding.sd_verify_feedback_ex(T, D, x, u, tau, want_acc_prob=False, want_status=False)
            names = ["accept_len", "tokens", "loss", "grad_draft"]
        elif kind == "errors":
            ws = torch.empty(binding.sd_workspace_bytes(B, k, V, binding._dtype_code(T)), dtype=torch.uint8, device="cuda")
            want = self.errors_with(binding, T, D, x, u, tau, ws)
            names = ["accept_len", "tokens", "loss", "error_grad", "status"]
        else:
            ws = torch.empty(binding.sd_greedy_workspace_bytes(B, k), dtype=torch.uint8, device="cuda")
            want = binding.sd_verify_greedy(T, x, workspace=ws)
            names = ["accept_len", "tokens", "argmax"]
        torch.cuda.synchronize()
        self.want = {n: getattr(want, n).clone() for n in names}
        self.out = want
        if kind == "step":
            self.fn = lambda: binding.sd_verify_feedback(T, D, x, u, tau, out=self.out)
        elif kind == "errors":
            self.fn = lambda: binding.sd_verify_error_feedback(T, D, x, u, tau, out=self.out)
        else:
            self.fn = lambda: binding.sd_verify_greedy(T, x, out=self.out)

    @staticmethod
    def errors_with(binding, T, D, x, u, tau, ws):
        """Error feedback on a caller workspace (the Python wrapper has none)."""
        B, k, V = D.shape
        o = binding.sd_verify_error_feedback(T, D, x, u, tau)        # output tensors of the right kinds
        rc = binding._lib.sd_verify_error_feedback(T.data_ptr(), D.data_ptr(), x.data_ptr(), u.data_ptr(), float(tau), B, k, V,
                                                   binding._dtype_code(T), o.accept_len.data_ptr(), o.tokens.data_ptr(),
                                                   o.loss.data_ptr(), o.error_grad.data_ptr(), o.status.data_ptr(), ws.data_ptr(),
                                                   ws.numel(), torch.cuda.current_stream().cuda_stream)
        assert rc == 0
        return o

    def forget(self):
        for n in self.want:
            getattr(self.out, n).fill_(-9)

    def check(self, what):
        torch.cuda.synchronize()
        for n, w in self.want.items():
            assert torch.equal(getattr(self.out, n), w), f"{what}: {n}"

    def run(self, what):
        self.forget()
        self.fn()
        self.check(what)

    def capture(self):
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            self.fn()
        return g


@pytest.mark.parametrize("kind", ["errors", "step", "greedy"])
@pytest.mark.parametrize("shape", [LARGE, SMALL])
def test_captured_calls_and_eager_calls_share_the_scratch(binding, kind, shape):
    call = Call(binding, kind, shape, 110)
    other = Call(binding, "step", SMALL if shape == LARGE else (40, 4, 8192, "f32"), 111)
    other.run("other, first")
    call.run("first")                  # grows the scratch to what it needs; its head is clean now
    call.run("second")
    other.run("other")
    call.run("third")
    graph = call.capture()             # captured on a clean head
    for turn in range(2):
        other.run("other, between")    # writes where `call` keeps its counters
        call.forget()
        graph.replay()
        call.check(f"replay {turn}")
        graph.replay()
        call.check(f"second replay {turn}")
        call.run(f"eager after replay {turn}")
        other.run("other, after")
    other.run("other")
    graph2 = call.capture()            # captured on a head that is not clean, and not run
    call.run("eager after a capture that was not run")
    call.forget()
    graph2.replay()
    call.check("replay of it")
    del graph, graph2


@pytest.mark.parametrize("shape", [LARGE, SMALL])
def test_error_feedback_after_a_wait_that_ran_out(binding, options, shape):
    """A kernel that gives up leaves tickets and its error flag behind: the next call of another kind on the
    library's scratch must not take them for its own.  (Nothing hangs: the waits simply run out.)"""
    call = Call(binding, "errors", shape, 112)
    late = Call(binding, "step", (64, 4, 8192, "f32"), 113)
    call.run("before")
    call.run("before, on a clean head")
    late.run("before")
    options(binding.SD_OPT_WAIT_POLLS, 4)
    late.fn()
    torch.cuda.synchronize()
    assert binding.sd_launch_info()["kernels"] == 1
    options(binding.SD_OPT_WAIT_POLLS, 1 << 21)
    call.run("after")
    call.run("after, once more")


def test_a_captured_call_keeps_its_scratch_when_a_larger_call_needs_more(binding):
    call = Call(binding, "step", SMALL, 114)
    larger = Call(binding, "step", (6000, 3, 512, "f32"), 115)      # more than the first buffer's 1 MiB
    binding.sd_release_cached_buffers()
    call.run("first")
    graph = call.capture()
    larger.run("larger")
    assert binding.sd_workspace_bytes(6000, 3, 512, 0) > 1 << 20
    fill = [torch.full((1 << 20,), 0xFF, dtype=torch.uint8, device="cuda") for _ in range(8)]   # would take freed memory over
    call.forget()
    graph.replay()
    call.check("replay on the buffer that was outgrown")
    larger.run("larger again")
    assert all(bool((f == 0xFF).all()) for f in fill)
    del graph


class EnsembleCall(Call):
    """An ensemble on the library's scratch (the Python wrapper brings its own), two learners."""

    def __init__(self, binding, shape, index):
        B, k, V, dtype = shape
        inp = synth.make_inputs(synth.custom_config(B=B, k=k, V=V, dtype=dtype, tau=0.9, index=index))
        T, D, _, _ = to_device(inp)
        Ds = [D, D.roll(1, 0).contiguous()]
        o = binding.sd_ensemble_feedback(T, Ds, inp.tau, 10.0, want_status=True)
        torch.cuda.synchronize()
        self.out = types.SimpleNamespace(loss=o.loss, grad0=o.grad[0], grad1=o.grad[1], round_loss=o.round_loss, cum_loss=o.cum_loss,
                                         weights=o.weights, status=o.status)
        self.want = {n: t.clone() for n, t in vars(self.out).items()}
        dptr, gptr = ((ctypes.c_void_p * 2)(*[t.data_ptr() for t in ts]) for ts in (Ds, o.grad))

        def fn(keep=(T, Ds, dptr, gptr)):
            rc = binding._lib.sd_ensemble_feedback(T.data_ptr(), dptr, 2, float(inp.tau), 10.0, B, k, V, binding._dtype_code(T), None,
                                                   o.loss.data_ptr(), gptr, o.round_loss.data_ptr(), o.cum_loss.data_ptr(),
                                                   o.weights.data_ptr(), o.status.data_ptr(), None, 0,
                                                   torch.cuda.current_stream().cuda_stream)
            assert rc == 0
        self.fn = fn


def test_a_held_ensemble_wants_no_scratch(binding):
    """Rows on the chip: nothing to allocate, so there need be none when the call is captured."""
    call = EnsembleCall(binding, (2, 3, 8192, "bf16"), 116)
    assert binding.sd_launch_info()["threads"] == 512
    call.run("eager")
    binding.sd_release_cached_buffers()
    graph = call.capture()
    call.forget()
    graph.replay()
    call.check("replay")
    del graph


def test_ensembles_and_other_calls_share_the_scratch(binding):
    """The ensemble's sweeps write where other calls keep words that must be zero, when they are issued and whenever a graph replays them."""
    call = EnsembleCall(binding, (60, 3, 20000, "bf16"), 117)
    assert binding.sd_launch_info()["threads"] == 256
    other = Call(binding, "step", LARGE, 118)
    call.run("first")
    other.run("other after an ensemble")
    call.run("second")
    other.run("other, again")
    graph = call.capture()
    assert binding.sd_launch_info()["threads"] == 256
    for turn in range(2):
        other.run("other, between")
        call.forget()
        graph.replay()
        call.check(f"replay {turn}")
        other.run("other after a replay")
        call.run("eager")
        other.run("other after both")
    del graph
