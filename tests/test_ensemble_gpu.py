"""GPU parity of the online-ensemble feedback (Sec. 3.3) against the CPU oracle: per-learner loss
and gradient within the tolerances of the single-draft step, the round's mean loss, the cumulative
losses and the Hedge weights.

Bars: loss |gpu - ref| <= tol*|ref| + 4e-7 with tol = 1e-5 (fp32 logits) / 2e-2 (bf16 logits);
gradient per row max|gpu - ref| <= tol*max|ref| + 8*2^-24*max(p,q)/tau; mean loss of the round and
cumulative loss like the loss; a weight is exp(-eps*cum)/Z, so its relative error is at most
2*eps times the absolute error of the cumulative losses, plus fp32 rounding of the stored weight.
"""
import numpy as np
import pytest
import torch

from oracle import sd_oracle
from paper_2603_12617_b200 import synth

pytestmark = pytest.mark.gpu

TOL = {"f32": 1e-5, "bf16": 2e-2}
LOSS_FLOOR = 4e-7
GRAD_FLOOR = 8 * 2.0 ** -24
EPS = 10.0


@pytest.fixture(scope="module")
def binding():
    import __graft_entry__ as entry
    entry.build()
    from paper_2603_12617_b200 import binding as b
    return b


def dev(a):
    t = torch.from_numpy(a).cuda()
    return t.view(torch.bfloat16) if a.dtype == np.uint16 else t


def f64(a):
    return (synth.bf16_bits_to_f32(a) if a.dtype == np.uint16 else a).astype(np.float64)


def pmax_of(z, tau):
    e = np.exp((z - z.max(axis=-1, keepdims=True)) / tau)
    return 1.0 / e.sum(axis=-1)


def compare(inp, Ds, out, ref, cum_in=None, eps=EPS, loss_floor=LOSS_FLOOR, grad_floor=GRAD_FLOOR):
    tol = TOL[inp.cfg.dtype]
    k = inp.cfg.k
    loss = out.loss.cpu().numpy().astype(np.float64)
    err = np.abs(loss - ref.loss)
    bound = tol * np.maximum(np.abs(ref.loss), 1e-6) + loss_floor
    assert (err <= bound).all(), f"loss: worst ratio {np.max(err / bound):.3g}"
    if out.grad is not None:
        pm = pmax_of(f64(inp.target_logits)[:, :k], inp.tau)
        for n, D in enumerate(Ds):
            g = out.grad[n].cpu().float().numpy().astype(np.float64)
            qm = pmax_of(f64(D), inp.tau)
            worst = np.abs(g - ref.grad[n]).max(axis=2)
            gb = tol * np.abs(ref.grad[n]).max(axis=2) + grad_floor * np.maximum(pm, qm) / inp.tau
            assert (worst <= gb).all(), f"grad of learner {n}: worst ratio {np.max(worst / gb):.3g}"
    rl = out.round_loss.cpu().numpy()
    cum = out.cum_loss.cpu().numpy()
    w = out.weights.cpu().numpy().astype(np.float64)
    lb = tol * np.maximum(np.abs(ref.round_loss), 1e-6) + loss_floor
    assert (np.abs(rl - ref.round_loss) <= lb).all()
    assert (np.abs(cum - ref.cum_loss) <= lb + 1e-15 * np.abs(ref.cum_loss)).all()
    assert abs(w.sum() - 1.0) < 1e-6
    assert (np.abs(w - ref.weights) <= 2 * eps * lb.max() * ref.weights + 2.0 ** -23).all(), (w, ref.weights)
    # the device's own weights are the exponential weighting of the device's own cumulative losses
    mine = np.exp(-eps * (cum - cum.min()))
    np.testing.assert_allclose(w, mine / mine.sum(), rtol=3e-7, atol=1e-12)


def run(binding, cfg, N=3, seqs=None, cum_in=None, want_grad=True, eps=EPS, **floors):
    inp = synth.make_inputs(cfg, sequences=seqs)
    Ds = synth.ensemble_drafts(inp, N)
    ref = sd_oracle.ensemble_feedback(inp.target_logits, Ds, inp.tau, eps, cum_loss=cum_in, want_grad=want_grad,
                                      nthreads=min(8, sd_oracle.max_threads()))
    cum_dev = None if cum_in is None else torch.from_numpy(np.asarray(cum_in, np.float64)).cuda()
    out = binding.sd_ensemble_feedback(dev(inp.target_logits), [dev(d) for d in Ds], inp.tau, eps,
                                       cum_loss=cum_dev, want_grad=want_grad, want_status=True)
    torch.cuda.synchronize()
    assert (out.status.cpu().numpy() == 0).all()
    compare(inp, Ds, out, ref, cum_in, eps, **floors)
    return inp, Ds, out, ref


@pytest.mark.parametrize("name,seqs", [("cfg1", None), ("cfg2", None), ("cfg3", range(0, 32, 11)),
                                       ("cfg4", range(2, 64, 23)), ("cfg5", range(0, 256, 97))])
def test_workloads_three_learners(binding, name, seqs):
    # the workloads at the contract's tolerance: no absolute term on the loss, no floor on the gradient
    run(binding, synth.CONFIGS[name], N=3, seqs=seqs, cum_in=[0.3, 0.1, 0.2], loss_floor=0.0, grad_floor=0.0)


@pytest.mark.parametrize("N", [1, 2, 5, 8])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_number_of_learners(binding, N, dtype):
    cfg = synth.custom_config(5, 3, 4096 + 8 * 37, dtype=dtype, tau=0.8, recipe="peaks")
    run(binding, cfg, N=N)


@pytest.mark.parametrize("B,k,V", [(1, 1, 8), (2, 1, 1024), (3, 4, 70000), (37, 2, 2048), (2, 64, 520)])
def test_shapes(binding, B, k, V):
    run(binding, synth.custom_config(B, k, V, dtype="f32"), N=3)
    run(binding, synth.custom_config(B, k, V, dtype="bf16"), N=2, want_grad=False)


@pytest.mark.parametrize("cluster", [1, 2, 3, 4, 6, 8])
def test_every_cluster_size(binding, cluster, options):
    options(binding.SD_OPT_CLUSTER, cluster)
    cfg = synth.custom_config(6, 3, 50000, dtype="f32", tau=0.9)
    run(binding, cfg, N=3)
    assert binding.sd_launch_info()["cluster_size"] == cluster


def test_each_learner_equals_the_single_draft_step_bit_for_bit(binding, options):
    """The units of the ensemble run the arithmetic of the single-draft step: at the same cluster
    size the same loss bits and the same gradient bits, whichever learner and wherever the unit
    falls in a cluster's range."""
    options(binding.SD_OPT_CLUSTER, 2)
    cfg = synth.CONFIGS["cfg2"]
    inp = synth.make_inputs(cfg)
    Ds = synth.ensemble_drafts(inp, 3)
    T = dev(inp.target_logits)
    x = torch.from_numpy(inp.draft_tokens).cuda()
    u = torch.from_numpy(inp.uniforms).cuda()
    out = binding.sd_ensemble_feedback(T, [dev(d) for d in Ds], inp.tau, EPS)
    for n, D in enumerate(Ds):
        one = binding.sd_verify_feedback(T, dev(D), x, u, inp.tau)
        torch.cuda.synchronize()
        assert torch.equal(one.loss, out.loss[n])
        assert torch.equal(one.grad_draft.view(torch.int16), out.grad[n].view(torch.int16))


def test_rounds_accumulate_in_place_and_weights_track_the_best_learner(binding):
    cfg = synth.custom_config(4, 3, 8192, dtype="bf16", tau=1.0)
    cum = torch.zeros(3, dtype=torch.float64, device="cuda")
    total = np.zeros(3)
    out = None
    for rnd in range(4):
        inp = synth.make_inputs(cfg, seed=synth.BASE_SEED + rnd)
        Ds = synth.ensemble_drafts(inp, 3, seed=synth.BASE_SEED + rnd)
        ref = sd_oracle.ensemble_feedback(inp.target_logits, Ds, inp.tau, EPS, cum_loss=total, want_grad=False)
        out = binding.sd_ensemble_feedback(dev(inp.target_logits), [dev(d) for d in Ds], inp.tau, EPS,
                                           cum_loss=cum, want_grad=False)
        torch.cuda.synchronize()
        total = ref.cum_loss
        cum = out.cum_loss                        # feeds the next round
        np.testing.assert_allclose(out.cum_loss.cpu().numpy(), total, rtol=1e-5)
    w = out.weights.cpu().numpy()
    assert w[0] > 0.99 or w.argmax() == int(np.argmin(total))


def test_refusals(binding):
    cfg = synth.custom_config(2, 2, 1001, dtype="f32")          # rows are not whole 16-byte vectors
    inp = synth.make_inputs(cfg)
    with pytest.raises(binding.SdVerifyError):
        binding.sd_ensemble_feedback(dev(inp.target_logits), [dev(inp.draft_logits)], 1.0, EPS)
    cfg = synth.custom_config(2, 2, 1024, dtype="f32")
    inp = synth.make_inputs(cfg)
    T, D = dev(inp.target_logits), dev(inp.draft_logits)
    with pytest.raises(binding.SdVerifyError):
        binding.sd_ensemble_feedback(T, [D] * 9, 1.0, EPS)        # more learners than SD_MAX_LEARNERS
    with pytest.raises(binding.SdVerifyError):
        binding.sd_ensemble_feedback(T, [D], 0.0, EPS)
    with pytest.raises(binding.SdVerifyError):
        binding.sd_ensemble_feedback(T, [D], 1.0, -1.0)
    # and the library still works afterwards
    out = binding.sd_ensemble_feedback(T, [D, T[:, :2].contiguous()], 1.0, EPS)
    torch.cuda.synchronize()
    assert float(out.round_loss[1]) < 1e-9 and float(out.weights[1]) > float(out.weights[0])


def test_full_size_bench_shape_equals_the_single_draft_step(binding, options):
    """The bench shape with 3 learners (B=256, k=6, V=128256, fp32; 62 units per cluster): every
    learner's loss and gradient bit-equal to the single-draft step on the same logits, and the
    weights from the device's own losses."""
    options(binding.SD_OPT_CLUSTER, 2)
    cfg = synth.CONFIGS["cfg5"]
    inp = synth.make_inputs(cfg)
    Ds = synth.ensemble_drafts(inp, 3)
    T = dev(inp.target_logits)
    x = torch.from_numpy(inp.draft_tokens).cuda()
    u = torch.from_numpy(inp.uniforms).cuda()
    dDs = [dev(d) for d in Ds]
    out = binding.sd_ensemble_feedback(T, dDs, inp.tau, EPS, want_status=True)
    torch.cuda.synchronize()
    assert (out.status.cpu().numpy() == 0).all()
    for n in range(3):
        one = binding.sd_verify_feedback(T, dDs[n], x, u, inp.tau)
        torch.cuda.synchronize()
        assert torch.equal(one.loss, out.loss[n])
        assert torch.equal(one.grad_draft, out.grad[n])
        del one
    mean = out.loss.double().mean(dim=(1, 2)).cpu().numpy()
    np.testing.assert_allclose(out.round_loss.cpu().numpy(), mean, rtol=1e-12)
    w = np.exp(-EPS * (mean - mean.min()))
    np.testing.assert_allclose(out.weights.cpu().numpy(), w / w.sum(), rtol=3e-7, atol=1e-12)


@pytest.mark.parametrize("lag,cluster", [(0, 2), (2, 1), (100, 3)])
def test_orders_of_the_walk_with_many_units_per_cluster(binding, lag, cluster, options):
    options(binding.SD_OPT_LAG, lag)
    options(binding.SD_OPT_CLUSTER, cluster)
    cfg = synth.custom_config(300, 4, 8192, dtype="bf16", tau=0.9, recipe="peaks")
    inp = synth.make_inputs(cfg)
    Ds = synth.ensemble_drafts(inp, 3)
    T = dev(inp.target_logits)
    x = torch.from_numpy(inp.draft_tokens).cuda()
    u = torch.from_numpy(inp.uniforms).cuda()
    dDs = [dev(d) for d in Ds]
    out = binding.sd_ensemble_feedback(T, dDs, inp.tau, EPS)
    for n in range(3):
        one = binding.sd_verify_feedback(T, dDs[n], x, u, inp.tau)
        torch.cuda.synchronize()
        assert torch.equal(one.loss, out.loss[n])
        assert torch.equal(one.grad_draft.view(torch.int16), out.grad[n].view(torch.int16))


def test_gradients_of_some_learners_can_be_left_out(binding):
    """A NULL entry in the array of gradient pointers: no gradient for that learner, the rest unchanged."""
    import ctypes
    cfg = synth.custom_config(4, 3, 8192, dtype="f32")
    inp = synth.make_inputs(cfg)
    Ds = synth.ensemble_drafts(inp, 3)
    T, dDs = dev(inp.target_logits), [dev(d) for d in Ds]
    full = binding.sd_ensemble_feedback(T, dDs, inp.tau, EPS)
    torch.cuda.synchronize()
    out = binding.EnsembleOutputs(loss=torch.empty_like(full.loss), grad=None,
                                  round_loss=torch.empty_like(full.round_loss), cum_loss=torch.empty_like(full.cum_loss),
                                  weights=torch.empty_like(full.weights), status=None)
    g0 = torch.full_like(full.grad[0], 7.0)
    g2 = torch.empty_like(full.grad[2])
    dptr = (ctypes.c_void_p * 3)(*[d.data_ptr() for d in dDs])
    gptr = (ctypes.c_void_p * 3)(None, None, g2.data_ptr())
    rc = binding._lib.sd_ensemble_feedback(T.data_ptr(), dptr, 3, float(inp.tau), EPS, cfg.B, cfg.k, cfg.V, 0, None,
                                           out.loss.data_ptr(), gptr, out.round_loss.data_ptr(),
                                           out.cum_loss.data_ptr(), out.weights.data_ptr(), None, None, 0, None)
    torch.cuda.synchronize()
    assert rc == 0
    assert torch.equal(out.loss, full.loss) and torch.equal(out.weights, full.weights)
    assert torch.equal(g2, full.grad[2]) and (g0 == 7.0).all()


# Two sweeps that share the target among the learners (csrc/sd_ensemble.cuh): bf16 rows of more than the chip holds twice.
@pytest.mark.parametrize("B,k,V,N", [(200, 3, 4104, 1), (1200, 2, 504, 3), (100, 3, 512 * 32 + 8, 2), (100, 3, 512 * 32 - 8, 2), (40, 3, 512 * 64 + 8, 3),
                                     (40, 4, 20000, 5), (30, 3, 30000, 8), (2, 64, 30000, 4), (2, 2, 5500008, 2)])
def test_two_sweeps(binding, options, B, k, V, N):
    """Rows shorter than a region, of a region more or less than an item, of the most items; one to four learners to a
    group, and groups of two sizes; with and without gradients; the cluster kernel, which one of its options selects."""
    cfg = synth.custom_config(B, k, V, dtype="bf16", tau=0.9)
    inp, Ds, out, ref = run(binding, cfg, N=N, cum_in=np.linspace(0.3, 0.1, N))
    info = binding.sd_launch_info()
    assert (info["path"], info["threads"], info["kernels"]) == (3, 256, 3 if N <= 4 else 5)
    T, dDs = dev(inp.target_logits), [dev(d) for d in Ds]
    cum = torch.from_numpy(np.linspace(0.3, 0.1, N)).cuda()
    only = binding.sd_ensemble_feedback(T, dDs, inp.tau, EPS, cum_loss=cum, want_grad=False)
    torch.cuda.synchronize()
    assert torch.equal(only.loss, out.loss) and torch.equal(only.weights, out.weights)
    options(binding.SD_OPT_CLUSTER, 2)
    other = binding.sd_ensemble_feedback(T, dDs, inp.tau, EPS, cum_loss=cum)
    assert binding.sd_launch_info()["threads"] == 1024
    torch.cuda.synchronize()
    compare(inp, Ds, other, ref, np.linspace(0.3, 0.1, N))


def test_two_sweeps_special_rows(binding):
    """Masked regions, entries far above all before them (target, one learner, both), identical models, a draft entry far
    below all others; and rows without a finite entry, which the status names."""
    B, k, V, N = 60, 3, 20000, 3
    inp = synth.make_inputs(synth.custom_config(B, k, V, dtype="bf16", tau=0.9, index=130))
    Ds = synth.ensemble_drafts(inp, N)
    T = inp.target_logits

    def value(v):
        return synth.f32_to_bf16_bits(np.array([v], np.float32))[0]
    ninf = np.uint16(0xFF80)
    T[0:2, :, 100:9000] = ninf
    for D in Ds:
        D[0:2, :, 100:6000] = ninf
    T[2, 0, 18000] = value(300)
    Ds[1][3, 1, 15000] = value(300)
    T[4, 1, 12000], Ds[2][4, 1, V - 3] = value(300), value(300)
    Ds[0][5] = T[5, :k]
    T[6, :, :V - 1] = ninf
    Ds[1][7, 2, 5] = value(-1e30)
    ref = sd_oracle.ensemble_feedback(T, Ds, inp.tau, EPS, nthreads=min(8, sd_oracle.max_threads()))
    out = binding.sd_ensemble_feedback(dev(T), [dev(d) for d in Ds], inp.tau, EPS, want_status=True)
    assert binding.sd_launch_info()["threads"] == 256
    torch.cuda.synchronize()
    assert (out.status.cpu().numpy() == 0).all()
    assert np.isfinite(ref.loss).all()
    compare(inp, Ds, out, ref)
    T[8, 1], Ds[2][9, 0] = ninf, ninf
    bad = binding.sd_ensemble_feedback(dev(T), [dev(d) for d in Ds], inp.tau, EPS, want_status=True)
    torch.cuda.synchronize()
    want = np.zeros(B)
    want[8:10] = binding.SD_STATUS_BAD_ROW
    assert (bad.status.cpu().numpy() == want).all()
    keep = [b for b in range(B) if b not in (8, 9)]
    assert torch.equal(bad.loss[:, keep], out.loss[:, keep])


def test_two_sweeps_keep_a_bad_draft_row_to_itself(binding):
    """A draft row without a finite entry -- of the first learner, whose constants the group takes the target's from, or of the
    last -- leaves everybody else's losses and gradients as they are, to the last bit."""
    B, k, V = 60, 3, 20000
    inp = synth.make_inputs(synth.custom_config(B, k, V, dtype="bf16", tau=0.9, index=135))
    for N in (3, 5):
        Ds = [dev(d) for d in synth.ensemble_drafts(inp, N)]
        T = dev(inp.target_logits)
        want = binding.sd_ensemble_feedback(T, Ds, inp.tau, EPS)
        torch.cuda.synchronize()
        bad = [(0, 9, 0), (N - 1, 20, 2)]
        for n, b, i in bad:
            Ds[n][b, i] = float("-inf")
        out = binding.sd_ensemble_feedback(T, Ds, inp.tau, EPS, want_status=True)
        assert binding.sd_launch_info()["threads"] == 256
        torch.cuda.synchronize()
        good = torch.ones(N, B, k, dtype=torch.bool, device="cuda")
        for n, b, i in bad:
            good[n, b, i] = False
        assert torch.equal(out.loss[good], want.loss[good])
        for n in range(N):
            assert torch.equal(out.grad[n][good[n]], want.grad[n][good[n]])
        assert [b for b in range(B) if out.status[b] != 0] == [9, 20] and (out.status[[9, 20]] == binding.SD_STATUS_BAD_ROW).all()


@pytest.mark.parametrize("N,left_out", [(3, (0, 1)), (3, (2,)), (5, (0, 4)), (5, (0, 1)), (5, (2, 3, 4)), (2, (0, 1))])
def test_two_sweeps_without_the_gradients_of_some_learners(binding, N, left_out):
    """Some of a group, a whole group (5 learners go as 2 and 3), all."""
    import ctypes
    cfg = synth.custom_config(60, 3, 20008, dtype="bf16", tau=0.9, index=136)
    inp = synth.make_inputs(cfg)
    T, Ds = dev(inp.target_logits), [dev(d) for d in synth.ensemble_drafts(inp, N)]
    full = binding.sd_ensemble_feedback(T, Ds, inp.tau, EPS)
    need = binding._lib.sd_ensemble_workspace_bytes(cfg.B, cfg.k, cfg.V, binding.SD_DTYPE_BF16, N)
    ws = torch.empty(need, dtype=torch.uint8, device="cuda")
    grads = [torch.full_like(g, 7.0) for g in full.grad]
    loss, small = torch.empty_like(full.loss), [torch.empty_like(t) for t in (full.round_loss, full.cum_loss, full.weights)]
    dptr = (ctypes.c_void_p * N)(*[d.data_ptr() for d in Ds])
    gptr = (ctypes.c_void_p * N)(*[None if n in left_out else g.data_ptr() for n, g in enumerate(grads)])
    rc = binding._lib.sd_ensemble_feedback(T.data_ptr(), dptr, N, float(inp.tau), EPS, cfg.B, cfg.k, cfg.V, binding.SD_DTYPE_BF16, None,
                                           loss.data_ptr(), gptr, *[t.data_ptr() for t in small], None, ws.data_ptr(), need, None)
    torch.cuda.synchronize()
    assert rc == 0 and binding.sd_launch_info()["threads"] == 256
    assert torch.equal(loss, full.loss) and torch.equal(small[2], full.weights)
    for n, g in enumerate(grads):
        assert (g == 7.0).all() if n in left_out else torch.equal(g, full.grad[n])


def test_two_sweeps_in_a_graph(binding):
    """A replay, whose scratch is the graph's, beside eager steps."""
    cfg = synth.custom_config(60, 3, 20000, dtype="bf16", tau=0.9, index=131)
    inp = synth.make_inputs(cfg)
    Ds = synth.ensemble_drafts(inp, 3)
    T, dDs = dev(inp.target_logits), [dev(d) for d in Ds]
    x, u = torch.from_numpy(inp.draft_tokens).cuda(), torch.from_numpy(inp.uniforms).cuda()
    want = binding.sd_ensemble_feedback(T, dDs, inp.tau, EPS)
    step = binding.sd_verify_feedback(T, dDs[0], x, u, inp.tau)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        out = binding.sd_ensemble_feedback(T, dDs, inp.tau, EPS)
        assert binding.sd_launch_info()["threads"] == 256
    for _ in range(2):
        g.replay()
        again = binding.sd_verify_feedback(T, dDs[0], x, u, inp.tau)
        torch.cuda.synchronize()
        assert torch.equal(again.tokens, step.tokens) and torch.equal(again.grad_draft, step.grad_draft)
        assert torch.equal(out.loss, want.loss) and torch.equal(out.weights, want.weights)
        assert all(torch.equal(a, b) for a, b in zip(out.grad, want.grad))


def test_two_sweeps_on_two_streams_at_once(binding):
    """Calls of the binding bring scratch of their own: they may overlap on the GPU."""
    cfg = synth.custom_config(60, 3, 20000, dtype="bf16", tau=0.9, index=132)
    inp = synth.make_inputs(cfg)
    Ds = synth.ensemble_drafts(inp, 3)
    T, dDs = dev(inp.target_logits), [dev(d) for d in Ds]
    want = [binding.sd_ensemble_feedback(T, list(d), inp.tau, EPS) for d in (dDs, dDs[::-1])]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    got = [[], []]
    for _ in range(6):
        for i, d in enumerate((dDs, dDs[::-1])):
            with torch.cuda.stream(streams[i]):
                got[i].append(binding.sd_ensemble_feedback(T, list(d), inp.tau, EPS))
                assert binding.sd_launch_info()["threads"] == 256
    torch.cuda.synchronize()
    for w, outs in zip(want, got):
        for o in outs:
            assert torch.equal(o.loss, w.loss) and torch.equal(o.weights, w.weights) and all(torch.equal(a, b) for a, b in zip(o.grad, w.grad))


def test_a_workspace_without_room_for_the_sweeps_takes_the_cluster_kernel(binding):
    """Callers that bring a flag word are served as before, and the library's own scratch takes the sweeps."""
    import ctypes
    cfg = synth.custom_config(60, 3, 20000, dtype="bf16", tau=0.9, index=133)
    inp = synth.make_inputs(cfg)
    Ds = synth.ensemble_drafts(inp, 3)
    T, dDs = dev(inp.target_logits), [dev(d) for d in Ds]
    want = binding.sd_ensemble_feedback(T, dDs, inp.tau, EPS)
    need = binding._lib.sd_ensemble_workspace_bytes(cfg.B, cfg.k, cfg.V, binding.SD_DTYPE_BF16, 3)
    dptr = (ctypes.c_void_p * 3)(*[d.data_ptr() for d in dDs])
    for nbytes, threads in ((256, 1024), (need - 256, 1024), (need, 256), (0, 256)):
        ws = torch.full((nbytes,), 0xA5, dtype=torch.uint8, device="cuda")
        loss = torch.empty_like(want.loss)
        small = [torch.empty(3, dtype=torch.float64, device="cuda") for _ in range(2)] + [torch.empty(3, device="cuda")]
        rc = binding._lib.sd_ensemble_feedback(T.data_ptr(), dptr, 3, float(inp.tau), EPS, cfg.B, cfg.k, cfg.V, binding.SD_DTYPE_BF16, None,
                                               loss.data_ptr(), None, *[t.data_ptr() for t in small], None,
                                               ws.data_ptr() if nbytes else None, nbytes, None)
        torch.cuda.synchronize()
        assert rc == 0 and binding.sd_launch_info()["threads"] == threads
        err = (loss - want.loss).abs()
        assert torch.equal(loss, want.loss) if threads == 256 else (err <= 1e-4 * want.loss.abs() + 4e-7).all()


def test_two_sweeps_count_their_kernels(binding):
    """No second sweep of a group of learners without a gradient; the first group's does the round in any case."""
    cfg = synth.custom_config(40, 3, 20000, dtype="bf16", tau=0.9, index=134)
    inp = synth.make_inputs(cfg)
    T, Ds = dev(inp.target_logits), [dev(d) for d in synth.ensemble_drafts(inp, 5)]
    for N, grad, kernels in ((4, True, 3), (4, False, 3), (5, True, 5), (5, False, 4)):
        binding.sd_ensemble_feedback(T, Ds[:N], inp.tau, EPS, want_grad=grad)
        info = binding.sd_launch_info()
        assert (info["threads"], info["kernels"]) == (256, kernels)
    torch.cuda.synchronize()
