"""The work that users of this framework give it, as cases that can be timed and compared.

Every case is one call (for the vocabulary-parallel step: the three calls) of a public entry point of
``paper_2603_12617_b200.binding`` on device tensors, as a serving loop makes it once per round.  The
sizes are those of the workloads in ``synth.CONFIGS`` and of the tests, and generic ones beside them;
the logits have the value structure of ``synth`` (a Gaussian or Zipf-shaped target, a draft that follows
it with noise, draft tokens drawn from the draft), made on the GPU from the seed.

``draw`` gives cases of the same ranges: 1 to 256 sequences, 1 to 8 draft tokens, vocabularies of
32 000 to 152 064 entries (whole 16-byte vectors for most, odd ones where the entry point takes
them), both element types, 2 to 4 learners, 2 to 8 shards, 64 to 1536 positions and 1024 to 4096
features for the output layer.
"""
from __future__ import annotations

import math

import torch

from paper_2603_12617_b200 import binding, shard

V_MIN, V_MAX = 32000, 152064
MAX_BYTES = 2_495_348_736          # the step on 256 sequences, 6 draft tokens, 128 256 fp32 entries
MAX_FLOPS = 2 * 1536 * 128256 * 4096
EPSILON = 10.0                     # learning rate of the Hedge weights in the paper's experiments


def _case(name, path, B, k, V, dtype, tau, values, **more):
    return {"name": name, "path": path, "B": B, "k": k, "V": V, "dtype": dtype, "tau": tau, "values": values, **more}


def listed():
    return [
        # One interactive user, the paper's own setting: latency of a single small call.
        _case("step B1 V32000 f32", "step", 1, 4, 32000, "f32", 1.0, "gauss", grad=True),
        # A few concurrent users of a small-vocabulary model.
        _case("step B8 V32000 bf16", "step", 8, 5, 32000, "bf16", 0.7, "peaks", grad=True),
        # Ordinary serving batches of large-vocabulary models, logits as the model head leaves them.
        _case("step B32 V128256 bf16", "step", 32, 8, 128256, "bf16", 1.0, "zipf", grad=True),
        _case("step B64 V151936 bf16", "step", 64, 4, 151936, "bf16", 0.8, "zipf_mixed", grad=True),
        # The largest batch, fp32 logits: the benchmark's default workload.
        _case("step B256 V128256 f32", "step", 256, 6, 128256, "f32", 1.0, "gauss", grad=True),
        # A vocabulary with an odd number of entries (tokens added, not padded): no 16-byte rows.
        _case("step B16 V50257 bf16", "step", 16, 5, 50257, "bf16", 1.0, "zipf", grad=True),
        # Greedy decoding, the mode of the paper's experiments: the target's argmax only.
        _case("greedy B32 V128256 bf16", "greedy", 32, 8, 128256, "bf16", 1.0, "zipf"),
        # Updates from the first wrong position only (OSD's feedback).
        _case("errors B64 V151936 bf16", "errors", 64, 4, 151936, "bf16", 0.8, "zipf_mixed"),
        # Optimistic updates: the step with the distance between last round's gradient and this one's.
        _case("hint B32 V128256 f32", "hint", 32, 6, 128256, "f32", 1.0, "gauss"),
        # An online ensemble of three draft heads against one target.
        _case("ensemble B32 V128256 bf16", "ensemble", 32, 8, 128256, "bf16", 1.0, "zipf", learners=3),
        # The weight gradient of the draft's output layer at the end of a round.
        _case("lmhead R1536 V128256", "lmhead", 256, 6, 128256, "bf16", 1.0, "gauss", features=4096),
        # One rank of a tensor-parallel output layer: its quarter of the vocabulary.
        _case("shard B64 V151936/4 bf16", "vp", 64, 4, 151936, "bf16", 0.8, "zipf_mixed", shards=4),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    path = rng.choice(["step"] * 6 + ["greedy"] * 2 + ["errors", "hint", "ensemble", "lmhead", "vp"])
    dtype = rng.choice(["f32", "bf16", "bf16"])
    V = rng.randint(V_MIN, V_MAX)
    ragged = path in ("step", "greedy") and rng.random() < 0.25
    V = V | 1 if ragged else V // 64 * 64 if rng.random() < 0.6 else V // 8 * 8
    c = {"path": path, "B": _log_int(rng, 1, 256), "k": rng.randint(1, 8), "V": V, "dtype": dtype,
         "tau": rng.choice([0.6, 0.7, 0.8, 1.0, 1.0, 1.2]), "values": rng.choice(["gauss", "peaks", "zipf", "zipf_mixed"])}
    if path == "step":
        c["grad"] = rng.random() < 0.85          # a round that does not update the draft asks for no gradient
    elif path == "ensemble":
        c["learners"] = rng.randint(2, 4)
    elif path == "vp":
        c["shards"] = rng.choice([2, 4, 8])
    elif path == "lmhead":
        c["dtype"] = "bf16"
        c["B"] = _log_int(rng, 8, 192)
        c["k"] = 8
        c["features"] = rng.choice([1024, 2048, 2560, 4096])
    while work(c)["bytes"] > MAX_BYTES or work(c)["flops"] > MAX_FLOPS:
        c["B"] = max(1, c["B"] * 3 // 4)
    return c


# ---- inputs ------------------------------------------------------------------------------------

def _normal(g, *shape):
    return torch.randn(shape, generator=g, device="cuda", dtype=torch.float32)


def _target(c, g):
    """Target logits [B,k+1,V] in fp32: a Gaussian body, with a few high peaks or a Zipf prior on top."""
    B, k, V, values = c["B"], c["k"], c["V"], c["values"]
    sigma = {"gauss": 2.0, "peaks": 3.0, "zipf": 2.5, "zipf_mixed": 2.0}[values]
    T = _normal(g, B, k + 1, V).mul_(sigma)
    if values == "peaks":
        at = torch.randint(0, V, (B, k + 1, 50), generator=g, device="cuda")
        T.scatter_add_(2, at, torch.full((B, k + 1, 50), 8.0, device="cuda"))
    elif values.startswith("zipf"):
        rank = torch.randperm(V, generator=g, device="cuda").float() + 1.0
        T -= rank.log_().mul_(1.1 if values == "zipf" else 1.0)
    return T


def _draft(c, g, T, scale):
    """A draft that follows the target's first k rows, with noise of `scale` times the usual size."""
    B, k, values = c["B"], c["k"], c["values"]
    D = _normal(g, B, k, c["V"])
    if values == "zipf_mixed":
        D *= torch.empty(B, 1, 1, device="cuda").uniform_(0.2, 3.0, generator=g)
    else:
        D *= {"gauss": 0.8, "peaks": 1.0, "zipf": 1.5}[values]
    D *= scale
    return D.add_(T[:, :k], alpha=0.8 if values == "zipf" else 1.0)


def prepare(case, seed):
    c = dict(case)
    g = torch.Generator(device="cuda").manual_seed(seed)
    dt = torch.float32 if c["dtype"] == "f32" else torch.bfloat16
    code = binding.SD_DTYPE_F32 if c["dtype"] == "f32" else binding.SD_DTYPE_BF16
    B, k, V = c["B"], c["k"], c["V"]
    if c["path"] == "lmhead":
        # gradients of logits: tiny nearly everywhere, a few large entries per position
        R = B * k
        grad = _normal(g, R, V).mul_(1e-3)
        at = torch.randint(0, V, (R, 3), generator=g, device="cuda")
        grad.scatter_add_(1, at, _normal(g, R, 3).mul_(0.3))
        c["grad_logits"] = grad.to(dt)
        c["hidden"] = _normal(g, R, c["features"]).to(dt)
        return c
    T32 = _target(c, g)
    c["T"] = T32.to(dt)
    if c["path"] == "greedy":
        # what a greedy draft proposes: the target's choice four times out of five
        best = T32[:, :k].argmax(2)
        other = torch.randint(0, V, (B, k), generator=g, device="cuda")
        agree = torch.rand(B, k, generator=g, device="cuda") < 0.8
        c["x"] = torch.where(agree, best, other).int()
        return c
    drafts = [_draft(c, g, T32, 2.0 ** n).to(dt) for n in range(c.get("learners", 1))]
    if c["path"] == "ensemble":
        c["drafts"] = drafts
        c["cum_loss"] = torch.rand(len(drafts), generator=g, device="cuda", dtype=torch.float64)
        return c
    D = c["D"] = drafts[0]
    c["x"] = torch.empty(B, k, dtype=torch.int32, device="cuda")
    for b in range(0, B, 32):      # 32 sequences at a time: the probabilities are a temporary
        q = torch.softmax(D[b:b + 32].float() / c["tau"], 2)
        c["x"][b:b + 32] = torch.multinomial(q.view(-1, V), 1, generator=g).view(-1, k).int()
    c["u"] = torch.randint(0, 1 << 24, (B, k + 1), generator=g, device="cuda").float() / (1 << 24)
    if c["path"] == "hint":
        # last round's gradient: a softmax difference of other logits of the same kind
        c["hint"] = (torch.softmax(D.float().roll(1, 2), 2) - torch.softmax(T32[:, :k].roll(1, 2), 2)).to(dt)
        c["ws"] = torch.empty(binding.sd_hint_workspace_bytes(B, k, V, code), dtype=torch.uint8, device="cuda")
    elif c["path"] == "vp":
        cuts = shard.vocab_cuts(V, c["shards"], c["T"].element_size())
        shards = [(c["T"][:, :, a:e].contiguous(), D[:, :, a:e].contiguous()) for a, e in cuts]
        spaces = [torch.empty(max(256, binding.sd_vp_workspace_bytes(B, k, e - a, code)), dtype=torch.uint8, device="cuda")
                  for a, e in cuts]
        # what the other ranks' gathers bring; this rank is the second one
        c["records"] = torch.stack([binding.sd_vp_partial(t, d, c["x"], c["tau"], a, V, w)
                                    for (t, d), (a, e), w in zip(shards, cuts, spaces)])
        masses = [binding.sd_vp_finish(t, d, c["x"], c["u"], c["tau"], a, V, c["records"], len(cuts), r, spaces[r],
                                       want_grad=False).local_mass
                  for r, ((t, d), (a, e)) in enumerate(zip(shards, cuts))]
        c["masses"] = torch.stack(masses)
        c["rank"], c["offset"], c["ws"] = 1, cuts[1][0], spaces[1]
        c["T"], c["D"] = shards[1]
    return c


def run(s):
    path = s["path"]
    if path == "step":
        o = binding.sd_verify_feedback(s["T"], s["D"], s["x"], s["u"], s["tau"], want_grad=s["grad"])
        return o.accept_len, o.tokens, o.loss, o.grad_draft
    if path == "greedy":
        o = binding.sd_verify_greedy(s["T"], s["x"])
        return o.accept_len, o.tokens, o.argmax
    if path == "errors":
        o = binding.sd_verify_error_feedback(s["T"], s["D"], s["x"], s["u"], s["tau"])
        return o.accept_len, o.tokens, o.loss, o.error_grad, o.status
    if path == "hint":
        o = binding.sd_verify_feedback_hint(s["T"], s["D"], s["x"], s["u"], s["tau"], s["hint"], workspace=s["ws"])
        return o.accept_len, o.tokens, o.loss, o.grad_draft, o.hint_err, o.status
    if path == "ensemble":
        o = binding.sd_ensemble_feedback(s["T"], s["drafts"], s["tau"], EPSILON, cum_loss=s["cum_loss"])
        return o.loss, o.grad, o.round_loss, o.cum_loss, o.weights
    if path == "lmhead":
        return binding.sd_lmhead_grad(s["grad_logits"], s["hidden"])
    # the three local calls of one rank; the gathers' results are in the state, this rank's records go
    # where its gather would put them
    G, r, V, off = s["shards"], s["rank"], s["V"], s["offset"]
    binding.sd_vp_partial(s["T"], s["D"], s["x"], s["tau"], off, V, s["ws"], out_records=s["records"][r])
    f = binding.sd_vp_finish(s["T"], s["D"], s["x"], s["u"], s["tau"], off, V, s["records"], G, r, s["ws"])
    tokens = binding.sd_vp_draw(s["T"], s["D"], s["x"], s["u"], s["tau"], off, V, f.accept_len, s["masses"], G, r,
                                f.status, s["ws"])
    return f.accept_len, f.loss, f.grad_shard, f.local_mass, f.status, tokens


# ---- what a pass cannot do without, and how exact its results are ---------------------------------

def work(case):
    B, k, V, path = case["B"], case["k"], case["V"], case["path"]
    e = 4 if case["dtype"] == "f32" else 2
    target, draft = B * (k + 1) * V * e, B * k * V * e
    small = B * (k + 1) * 16
    if path == "lmhead":
        R, d = B * k, case["features"]
        return {"bytes": R * (V + d) * 2 + V * d * 4, "flops": 2 * R * V * d}
    if path == "greedy":
        return {"bytes": target + small, "flops": B * (k + 1) * V}
    pairs = B * k * V
    if path == "errors":
        return {"bytes": target + draft + B * V * e + small, "flops": 10 * pairs}
    if path == "ensemble":
        n = case["learners"]
        return {"bytes": draft + 2 * n * draft + n * small, "flops": 20 * n * pairs}
    if path == "vp":
        target, draft, pairs = target // case["shards"], draft // case["shards"], pairs // case["shards"]
        return {"bytes": target + 2 * draft + small, "flops": 20 * pairs}
    if path == "hint":
        return {"bytes": target + 3 * draft + small, "flops": 23 * pairs}
    return {"bytes": target + (2 if case["grad"] else 1) * draft + small, "flops": 20 * pairs}


def tolerance(case):
    # Measured against the same results in 64-bit arithmetic and stated at about four times that: fp32
    # gradients and losses are off by up to 3e-7 (more where draft and target nearly agree and p - q
    # cancels), bf16 gradients by their rounding (1.7e-3, at most 3.9e-3 of a value), the fp32 sums of the
    # matrix product by 1.7e-6 (largest 1.7e-5 of the root mean square).
    # "differ": a uniform that falls within rounding of a threshold or of a cumulative sum may go either way.
    if case["path"] == "greedy":
        return "exact"
    if case["path"] == "lmhead":
        return {"rel": 7e-6, "max": 7e-5}
    if case["dtype"] == "f32":
        return {"rel": 2e-6, "max": 1e-4, "differ": 0.004}
    return {"rel": 7e-3, "max": 1.6e-2, "differ": 0.004}
