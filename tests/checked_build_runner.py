"""Runs every entry point on tiny, ragged and multi-stage shapes, on every kernel that it may take, through whichever build of the
library SD_VERIFY_LIBRARY names, compares with the CPU oracle, and prints what sd_bounds_report counted.
Started as a child process by test_bounds_checked_gpu.py (the library is chosen at import)."""
import json
import sys

import numpy as np
import torch

from oracle import sd_oracle
from paper_2603_12617_b200 import binding as b, shard, synth
from test_parity_gpu import check, oracle_of, to_device


def shifted(t, lead):
    """The tensor's values `lead` elements past a 16-byte boundary."""
    buf = torch.empty(t.numel() + lead, dtype=t.dtype, device=t.device)
    v = buf[lead:].view(t.shape)
    v.copy_(t)
    return v


# Which kernel a call took, by its threads a block; the error-position feedback's second one has 256 in any case.
KERNEL = {1024: "cluster", 512: "held", 256: "sweeps"}
SEEN = set()


def took(entry, sweeps=3):
    info = b.sd_launch_info()
    kernel = "element-wise" if info["path"] == 0 else KERNEL[info["threads"]]
    assert info["kernels"] == {"sweeps": sweeps}.get(kernel, 2 if entry in ("errors", "ensemble") else 1), (entry, info)
    SEEN.add((entry, kernel))
    return kernel


def sharded(T, D, x, u, tau, cuts):
    """The vocabulary-parallel step, every rank's calls."""
    B, k, V = D.shape
    code, G = (b.SD_DTYPE_F32 if T.dtype == torch.float32 else b.SD_DTYPE_BF16), len(cuts)
    Ts = [T[:, :, a:c].contiguous() for a, c in cuts]
    Ds = [D[:, :, a:c].contiguous() for a, c in cuts]
    ws = [torch.empty(max(256, b.sd_vp_workspace_bytes(B, k, c - a, code)), dtype=torch.uint8, device="cuda") for a, c in cuts]
    recs = torch.stack([b.sd_vp_partial(Ts[r], Ds[r], x, tau, cuts[r][0], V, ws[r]) for r in range(G)], 0).contiguous()
    fins = [b.sd_vp_finish(Ts[r], Ds[r], x, u, tau, cuts[r][0], V, recs, G, r, ws[r]) for r in range(G)]
    m = torch.stack([f.local_mass for f in fins], 0).contiguous()
    tokens = torch.stack([b.sd_vp_draw(Ts[r], Ds[r], x, u, tau, cuts[r][0], V, fins[r].accept_len, m, G, r, fins[r].status, ws[r])
                          for r in range(G)], 0).max(0).values
    return fins[0].accept_len, tokens


def main():
    assert b.sd_bounds_report() is not None, "this build of the library has no range checks"
    shapes = [(2, 2, 5, "f32"), (3, 1, 17, "bf16"), (2, 3, 1023, "f32"), (4, 2, 1024, "bf16"), (5, 3, 7168 + 256, "f32"),
              (3, 2, 50000, "bf16"), (9, 3, 65536, "f32"), (2, 64, 520, "f32"), (40, 2, 16392, "bf16")]
    for (B, k, V, dt) in shapes:
        cfg = synth.custom_config(B, k, V, dtype=dt, tau=0.9, index=90)
        inp = synth.make_inputs(cfg)
        T, D, x, u = to_device(inp)
        ref = oracle_of(inp)
        es = T.element_size()
        whole = (V * es) % 16 == 0
        for cluster in (0, 3, 8):
            b.sd_set_option(b.SD_OPT_CLUSTER, cluster)
            ex = b.sd_verify_feedback_ex(T, D, x, u, inp.tau)
            kernel = took("step")
            assert not whole or (kernel == "cluster") == (cluster != 0)
            check(inp, ex, ref, max_band_frac=1.0)
            h = b.sd_verify_feedback_hint(T, D, x, u, inp.tau, torch.zeros_like(D))
            assert took("hint") == kernel or not whole
            check(inp, h, ref, max_band_frac=1.0)
            if whole:
                e = b.sd_verify_error_feedback(T, D, x, u, inp.tau)
                assert took("errors") == kernel
                assert torch.equal(e.accept_len, h.accept_len)
                n = e.accept_len.long()
                rows = torch.where((n < k)[:, None], ex.grad_draft[torch.arange(B, device="cuda"), n.clamp(max=k - 1)], 0)
                assert torch.equal(e.error_grad, rows)
                m = b.sd_ensemble_feedback(T, [D, D.clone()], inp.tau, 10.0)
                took("ensemble")
                assert (m.loss - ex.loss).abs().max() <= 1e-4 * ex.loss.abs().max() + 4e-7 and torch.equal(m.loss[0], m.loss[1])
        b.sd_set_option(b.SD_OPT_CLUSTER, 0)
        check(inp, b.sd_verify_feedback(T, D, x, u, inp.tau), ref, max_band_frac=1.0)
        g = b.sd_verify_greedy(T, x)
        gref = sd_oracle.verify_greedy(inp.target_logits, inp.draft_tokens)
        assert (g.accept_len.cpu().numpy() == gref.accept_len).all() and (g.tokens.cpu().numpy() == gref.tokens).all()
        if whole and V // (16 // es) >= 2:
            sharded(T, D, x, u, inp.tau, [(0, V // 2 // (16 // es) * (16 // es)), (V // 2 // (16 // es) * (16 // es), V)])
        torch.cuda.synchronize()

    # the two sweeps: whole-vector rows of more than fit the chip at once, odd rows wherever they start
    for (B, k, V, dt, leadT, leadD) in [(40, 3, 58000, "bf16", 0, 0), (24, 3, 72004, "f32", 0, 0), (1300, 2, 4104, "bf16", 0, 0), (1300, 2, 504, "bf16", 0, 0),
                                        (200, 2, 4097, "bf16", 1, 6), (150, 3, 2051, "f32", 2, 1), (3, 2, 50257, "bf16", 0, 0),
                                        (2, 2, 512 * 65 - 1, "bf16", 3, 0), (3, 2, 40003, "f32", 3, 3)]:
        cfg = synth.custom_config(B, k, V, dtype=dt, tau=0.9, index=91)
        inp = synth.make_inputs(cfg)
        T, D, x, u = to_device(inp)
        T, D = shifted(T, leadT), shifted(D, leadD)
        out = b.StepOutputs(accept_len=torch.empty(B, dtype=torch.int32, device="cuda"),
                            tokens=torch.empty((B, k + 1), dtype=torch.int32, device="cuda"),
                            loss=torch.empty((B, k), device="cuda"), grad_draft=shifted(torch.zeros_like(D), leadD),
                            acc_prob=torch.empty((B, k), device="cuda"), status=torch.empty(B, dtype=torch.int32, device="cuda"))
        b.sd_verify_feedback_ex(T, D, x, u, inp.tau, out=out)
        assert took("step") == "sweeps"
        check(inp, out, oracle_of(inp), max_band_frac=1.0)
        only = b.sd_verify_feedback(T, D, x, u, inp.tau, want_loss=False, want_grad=False)
        assert torch.equal(only.tokens, out.tokens)
        if V * T.element_size() % 16 == 0:
            e = b.sd_verify_error_feedback(T, D, x, u, inp.tau)
            assert took("errors") == "sweeps"
            h = b.sd_verify_feedback_hint(T, D, x, u, inp.tau, torch.zeros_like(D))
            assert took("hint") == "sweeps"
            assert torch.equal(e.tokens, out.tokens) and torch.equal(h.tokens, out.tokens)
        if dt == "bf16" and V % 8 == 0:
            # (one and two groups of learners; sums of another order than the step's, so its values to rounding)
            for N, grad in ((2, True), (4, False), (5, True), (5, False)):
                m = b.sd_ensemble_feedback(T, [D.roll(n, 0) for n in range(N)], inp.tau, 10.0, want_grad=grad)
                assert took("ensemble", 3 if N <= 4 else 5 if grad else 4) == "sweeps"
                assert ((m.loss[0] - out.loss).abs() <= 1e-5 * out.loss + 4e-7).all()
                if grad:
                    assert ((m.grad[0].float() - out.grad_draft.float()).abs() <= 2.0 ** -7 * out.grad_draft.float().abs() + 1e-6).all()
        torch.cuda.synchronize()

    # the sharded step with regions one and two at a time, and with both sizes of the draw's blocks
    for (B, k, V, dt, cut) in [(700, 1, 256 * 13, "f32", 256 * 7), (400, 2, 256 * 52, "f32", 256 * 26 + 4), (600, 2, 512 * 3 + 8, "bf16", 512), (4, 2, 512 * 300, "bf16", 512 * 170)]:
        inp = synth.make_inputs(synth.custom_config(B, k, V, dtype=dt, tau=0.9, index=92))
        T, D, x, u = to_device(inp)
        accept_len, tokens = sharded(T, D, x, u, inp.tau, [(0, cut), (cut, V)])
        ref = oracle_of(inp)
        safe = (ref.accept_band.sum(1) == 0) & (ref.cdf_margin > 1e-6)
        assert (accept_len.cpu().numpy() == ref.accept_len)[safe].all() and (tokens.cpu().numpy() == ref.tokens)[safe].all()
    # a later rule may not take a kernel out of this run
    assert SEEN == {(e, n) for e in ("step", "hint", "errors", "ensemble") for n in ("cluster", "held", "sweeps")} \
        | {("step", "element-wise"), ("hint", "element-wise")}, SEEN
    print("REPORT " + json.dumps(b.sd_bounds_report()))


if __name__ == "__main__":
    sys.exit(main())
