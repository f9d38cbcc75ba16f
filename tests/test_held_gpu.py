"""The kernel that holds the logits in registers (csrc/sd_held.cuh) at the sizes where its cuts can go wrong -- one
vector, a region more or less than a cluster's warps take, its largest clusters, as many units as are
resident -- and on special rows, against the oracle, with the calls that share it."""
import numpy as np
import pytest
import torch

from oracle import sd_oracle
from paper_2603_12617_b200 import synth
from test_parity_gpu import check, check_hint_error, hint_of, oracle_of, to_device

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def binding():
    import __graft_entry__ as entry
    entry.build()
    from paper_2603_12617_b200 import binding as b
    return b


def alike(binding, Td, Dd, xd, ud, tau, ex):
    """The step without gradient and the error-position feedback take the same decisions as the step."""
    B, k = xd.shape
    plain = binding.sd_verify_feedback(Td, Dd, xd, ud, tau, want_loss=False, want_grad=False)
    err = binding.sd_verify_error_feedback(Td, Dd, xd, ud, tau)
    assert binding.sd_launch_info()["kernels"] == 2
    torch.cuda.synchronize()
    for o in (plain, err):
        assert torch.equal(o.accept_len, ex.accept_len) and torch.equal(o.tokens, ex.tokens)
    assert torch.equal(err.status, ex.status)
    n = ex.accept_len.long()
    rows = torch.where((n < k)[:, None], ex.grad_draft[torch.arange(B, device="cuda"), n.clamp(max=k - 1)], 0)
    return err, rows


# A region is 64 vectors (256 fp32 or 512 bf16 entries), a cluster up to 16 blocks of 16 warps with up to 4 regions each.
@pytest.mark.parametrize("B,k,V,dtype", [
    (1, 1, 4, "f32"), (49, 2, 256 * 16, "f32"), (3, 3, 256 * 16 + 4, "f32"), (2, 2, 256 * 256, "f32"), (2, 2, 256 * 256 + 4, "f32"),
    (2, 1, 256 * 769, "f32"), (1, 64, 256 * 17 - 4, "f32"), (2, 3, 520, "bf16"), (49, 2, 512 * 15 + 8, "bf16"), (8, 5, 32000, "bf16"),
    (2, 2, 512 * 256 - 8, "bf16"), (4, 5, 128256, "bf16"), (1, 4, 152064, "bf16")])
def test_held_rows_match_the_oracle(binding, B, k, V, dtype):
    inp = synth.make_inputs(synth.custom_config(B=B, k=k, V=V, dtype=dtype, tau=0.9, index=130))
    T, D, x, u = to_device(inp)
    ref = oracle_of(inp)
    ex = binding.sd_verify_feedback_ex(T, D, x, u, inp.tau)
    info = binding.sd_launch_info()
    assert (info["path"], info["kernels"], info["threads"]) == (1, 1, 512)
    check(inp, ex, ref, max_band_frac=1.0)
    err, rows = alike(binding, T, D, x, u, inp.tau, ex)
    assert torch.equal(err.loss, ex.loss) and torch.equal(err.error_grad, rows)
    bits = hint_of(inp, synth.BASE_SEED + 31)
    H = torch.from_numpy(bits).cuda()
    H = H.view(torch.bfloat16) if dtype == "bf16" else H
    hint = binding.sd_verify_feedback_hint(T, D, x, u, inp.tau, H, grad_out=H)
    ens = binding.sd_ensemble_feedback(T, [D], inp.tau, 10.0)
    torch.cuda.synchronize()
    assert torch.equal(hint.grad_draft, ex.grad_draft) and torch.equal(hint.tokens, ex.tokens) and torch.equal(hint.loss, ex.loss)
    if V > 512:      # (a hint error of nearly nothing has no relative bar)
        check_hint_error(inp, bits, hint.hint_err.cpu().numpy(), 2e-4 if dtype == "f32" else 1e-3)
    one = sd_oracle.ensemble_feedback(inp.target_logits, [inp.draft_logits], inp.tau, 10.0, want_grad=False)
    np.testing.assert_allclose(ens.loss.cpu().numpy(), one.loss, rtol=1e-5 if dtype == "f32" else 2e-2, atol=4e-7)
    tol = 1e-5 if dtype == "f32" else 2e-2
    assert (ens.grad[0].float() - ex.grad_draft.float()).abs().max() <= tol * ex.grad_draft.float().abs().max()


@pytest.mark.parametrize("k,V,dtype", [(2, 5000, "bf16"), (3, 7204, "f32"), (1, 512 * 16 - 8, "bf16")])
def test_special_rows(binding, k, V, dtype):
    B = 16
    inp = synth.make_inputs(synth.custom_config(B=B, k=k, V=V, dtype=dtype, tau=0.9, index=131))
    T, D, x = inp.target_logits, inp.draft_logits, inp.draft_tokens

    def value(v):
        return np.float32(v) if dtype == "f32" else synth.f32_to_bf16_bits(np.array([v], np.float32))[0]
    ninf = value(-np.inf)
    half, last = V // 2, k - 1
    T[0:2, :, 100:half] = ninf                     # whole regions masked, in the target further than in the draft
    D[0:2, :, 100:V // 3] = ninf
    x[0:2] = np.clip(x[0:2], half, None)
    x[1, 0] = half - 5                             # p(x) = 0, q(x) > 0: rejected
    T[2, 0, int(0.9 * V)] = value(300)             # far above everything else: target only,
    D[3, last, int(0.75 * V)] = value(300)         # draft only,
    T[4, k, V - 1] = value(300)                    # the bonus row's last entry
    D[5] = T[5, :k]                                # identical models
    D[6, 0, 5] = ninf                              # q = 0 where p > 0: infinite divergence
    x[6, 0] = 7
    x[7, last] = V                                 # tokens outside the vocabulary
    x[8, 0] = -3
    T[9], D[9], x[9, last] = 0, 0, V + 5           # a rejection without residual mass: draw from p
    T[10, 0], D[11, last] = ninf, ninf             # rows without a finite entry
    T[12, :, :V - 1] = ninf                        # one finite entry, the row's last
    T[13, 0, 0], D[14, 0, 9] = value(np.nan), value(np.inf)
    unspecified = [10, 11, 13, 14]
    good = [b for b in range(B) if b not in unspecified]
    Td, Dd, xd, ud = to_device(inp)
    out = binding.sd_verify_feedback_ex(Td, Dd, xd, ud, inp.tau)
    assert binding.sd_launch_info()["threads"] == 512
    torch.cuda.synchronize()
    ref = oracle_of(inp, good)
    assert ref.status[good.index(9)] == 5 and ref.accept_len[good.index(9)] == last and ref.accept_len[good.index(1)] == 0
    check(inp, out, ref, seqs=good, max_band_frac=1.0)
    assert out.loss[5].abs().max() == 0 and out.accept_len[5] == k and torch.isinf(out.loss[6, 0])
    st, n, tok = out.status.cpu().numpy(), out.accept_len.cpu().numpy(), out.tokens.cpu().numpy()
    for b in unspecified:
        assert st[b] & binding.SD_STATUS_BAD_ROW
        assert 0 <= n[b] <= k and 0 <= tok[b, n[b]] < V and (tok[b, n[b] + 1:] == -1).all()
    err, rows = alike(binding, Td, Dd, xd, ud, inp.tau, out)
    assert torch.equal(err.loss[good], out.loss[good]) and torch.equal(err.error_grad[good], rows[good])


@pytest.mark.parametrize("V,dtype", [(520, "f32"), (256 * 17 - 4, "f32"), (256 * 16 * 4, "f32"), (520, "bf16"), (32000, "bf16")])
@pytest.mark.parametrize("tau", [2e29, 1e30, 1e33])
def test_nothing_behind_the_end_of_a_row_takes_part(binding, V, dtype, tau):
    """So hot that every probability is 1/V to fp32 (logits over the temperature are far below 2^-24): a draw with uniform u is
    entry u V, off by one at most for the rounding of fp32 sums of equal terms, whether it comes from a bonus row or
    from a rejection without residual mass; whatever lies behind the row's last entry must have no share in it."""
    B, k = 24, 2
    inp = synth.make_inputs(synth.custom_config(B=B, k=k, V=V, dtype=dtype, tau=1.0, index=132))
    inp.uniforms[:, k] = (np.arange(B) + 0.5).astype(np.float32) / B
    inp.draft_tokens[1::2, 1] = V                  # every second sequence: rejected there
    T, D, x, u = to_device(inp)
    ex = binding.sd_verify_feedback_ex(T, D, x, u, tau)
    assert binding.sd_launch_info()["threads"] == 512
    alike(binding, T, D, x, u, tau, ex)
    hint = binding.sd_verify_feedback_hint(T, D, x, u, tau, torch.zeros_like(D))
    torch.cuda.synchronize()
    want = torch.tensor([k, 1] * (B // 2), dtype=torch.int32, device="cuda")
    for o in (ex, hint):
        assert torch.equal(o.accept_len, want)
        assert (o.tokens.gather(1, want[:, None].long()).squeeze(1) - u[:, k] * V).abs().max() <= 1
        assert (o.loss.abs() <= 1e-6).all() and (o.grad_draft.float().abs() * tau * V <= 1e-6).all()


def small_workspace(binding, T, k, hint=False):
    """Without room for the two sweeps: two rounds of held rows are the faster way then."""
    B, V = T.shape[0], T.shape[2]
    size = (binding.sd_hint_workspace_bytes if hint else binding.sd_workspace_bytes)(B, k, V, binding._dtype_code(T))
    return torch.full((size - 256,), 0xA5, dtype=torch.uint8, device="cuda")


def errors_in(binding, T, D, x, u, tau, ws):
    B, k = x.shape
    o = binding.ErrorFeedbackOutputs(torch.empty(B, dtype=torch.int32, device="cuda"), torch.empty(B, k + 1, dtype=torch.int32, device="cuda"),
                                     torch.empty(B, k, device="cuda"), torch.empty_like(D[:, 0]), torch.empty(B, dtype=torch.int32, device="cuda"))
    p = [t.data_ptr() for t in (T, D, x, u)]
    rc = binding._lib.sd_verify_error_feedback(*p, tau, B, k, T.shape[2], binding._dtype_code(T), o.accept_len.data_ptr(), o.tokens.data_ptr(),
                                               o.loss.data_ptr(), o.error_grad.data_ptr(), o.status.data_ptr(), ws.data_ptr(), ws.numel(),
                                               torch.cuda.current_stream().cuda_stream)
    assert rc == 0
    return o


# Clusters of 1, 3 and 4 blocks.  B = 0: as many sequences as clusters of three are resident, with one draft token two rounds exactly,
# in which the drawn rows fit no shape of one round of their own (one cluster of such a size is held back) and take that of the first pass.
@pytest.mark.parametrize("B,k,V,dtype", [(60, 3, 512 * 64 - 8, "bf16"), (50, 4, 256 * 64, "f32"), (15, 4, 512 * 180 + 8, "bf16"),
                                         (0, 1, 512 * 180 - 8, "bf16"), (12, 4, 256 * 256 - 4, "f32")])
def test_two_rounds(binding, B, k, V, dtype):
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    for n in range(74, 37, -1) if B == 0 else []:
        Z = torch.zeros(n, k + 1, V, dtype=dt, device="cuda")
        binding.sd_verify_feedback_ex(Z, Z[:, :k].contiguous(), torch.zeros(n, k, dtype=torch.int32, device="cuda"),
                                      torch.zeros(n, k + 1, device="cuda"), 1.0, workspace=small_workspace(binding, Z, k))
        if binding.sd_launch_info()["threads"] == 512:
            B = n
            break
    inp = synth.make_inputs(synth.custom_config(B=B, k=k, V=V, dtype=dtype, tau=0.9, index=133))
    T, D, x, u = to_device(inp)
    C = -(-V // (512 if dtype == "bf16" else 256) // 64)
    resident = torch.cuda.get_device_properties(0).multi_processor_count // C
    assert resident < B * (k + 1) <= 2 * resident
    ex = binding.sd_verify_feedback_ex(T, D, x, u, inp.tau, workspace=small_workspace(binding, T, k))
    info = binding.sd_launch_info()
    assert (info["path"], info["kernels"], info["threads"], info["cluster_size"], info["blocks"]) == (1, 1, 512, C, C * B * (k + 1))
    check(inp, ex, oracle_of(inp), max_band_frac=1.0)
    err = errors_in(binding, T, D, x, u, inp.tau, small_workspace(binding, T, k))
    info = binding.sd_launch_info()
    assert (info["path"], info["kernels"], info["threads"]) == (4, 2, 512) and (k > 1 or (info["cluster_size"], info["blocks"]) == (C, C * B))
    hint = binding.sd_verify_feedback_hint(T, D, x, u, inp.tau, torch.zeros_like(D), workspace=small_workspace(binding, T, k, hint=True))
    assert binding.sd_launch_info()["blocks"] == C * B * (k + 1)
    ens = binding.sd_ensemble_feedback(T, [D], inp.tau, 10.0)
    torch.cuda.synchronize()
    for o in (err, hint):
        assert torch.equal(o.accept_len, ex.accept_len) and torch.equal(o.tokens, ex.tokens) and torch.equal(o.loss, ex.loss)
        assert torch.equal(o.status, ex.status)
    n = ex.accept_len.long()
    assert torch.equal(err.error_grad, torch.where((n < k)[:, None], ex.grad_draft[torch.arange(B, device="cuda"), n.clamp(max=k - 1)], 0))
    assert torch.equal(hint.grad_draft, ex.grad_draft) and torch.equal(ens.loss[0], ex.loss) and torch.equal(ens.grad[0], ex.grad_draft)
