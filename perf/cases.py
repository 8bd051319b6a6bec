"""The work that programs built on this framework ask of it, as cases that can be timed.

A case is one pass through the public entry points (``PruneContext.prune_step``, and the stage calls as
``tensor_parallel.prune_step_head_sharded`` strings them together) on inputs that are on the GPU already:

* ``frame``    a robot's control loop: one camera frame, one prune point, a fresh episode on every pass;
* ``batch``    a server: a ragged batch of requests, descriptors handed over as the plain list that changes with
               every batch;
* ``episode``  the action iteration: several steps of one episode, scores carried over, the first one a cold start;
               with ``reuse`` the program says which rows changed and the logits of the others are reused;
* ``requests`` independent single-frame requests in flight beside one another (``FLAG_INPUTS_STABLE``);
* ``patch``    Alg. 1 patch by patch, alone or batched;
* ``shard``    one rank of a head-sharded server: scores, selection and row copy as calls of their own.

Inputs follow the repository's synthetic recipe (``workloads``: hidden ~ N(0, 1), salient rows scaled, projections by
random weights, everything rounded once), drawn on the GPU.  Output buffers are the program's own and zero where
nothing is written, so they are returned whole.
"""
import random

import torch

from paper_2604_09244_b200 import mvla, tensor_parallel
from paper_2604_09244_b200.workloads import Sample, layout_2d_3d_txt

_7B = {"d_model": 4096, "heads": 32, "head_dim": 128}     # LLaMA-2-7B width: the paper's host model


def _case(kind, **kw):
    c = {"kind": kind, "dtype": "bf16", "batch": 1, "txt_lo": 32, "txt_hi": 32, "n_2d": 256, "n_3d": 512,
         "kv_heads": 0, "mode": "adaptive", "keep_lo": 0.3, "keep_hi": 0.3, "keep_2d": 0.4, "keep_3d": 0.3,
         "steps": 1, "requests": 1, "reuse": False, "text_first": False, "shape": 0}
    c.update(_7B)
    c.update(kw)
    return c


def listed():
    return [
        # The reference-sized problem of configs[0]: what a developer's check or a small policy runs; all latency.
        _case("frame", name="tiny_fp32", dtype="fp32", d_model=512, heads=8, head_dim=64, txt_lo=16, txt_hi=16, n_2d=64,
              n_3d=128, keep_lo=0.5, keep_hi=0.5),
        # One camera frame of a 7B policy (configs[1], the benchmark's default): fixed keep ratios per modality.
        _case("frame", name="frame_7b", mode="fixed"),
        # The same frame in a quantised deployment: e4m3 q / k / v, four query heads to a key head.
        _case("frame", name="frame_fp8_grouped", dtype="fp8", kv_heads=8),
        # Three cameras and a dense point cloud (configs[2], first prune point), odd sizes of text and cloud.
        _case("frame", name="multi_view", txt_lo=47, txt_hi=47, n_2d=768, n_3d=1023, keep_lo=0.25, keep_hi=0.25),
        # Batched serving (configs[3]): 16 requests, ragged text, every request with a keep ratio of its own.
        _case("batch", name="batch_16", batch=16, txt_lo=16, txt_hi=64, keep_lo=0.2, keep_hi=0.6),
        # The largest: eight robots with six cameras and a large cloud each, more tokens than most deployments have.
        _case("batch", name="batch_8_six_views", batch=8, txt_lo=48, txt_hi=64, n_2d=1536, n_3d=2048, keep_lo=0.2,
              keep_hi=0.3),
        # Eight action steps of one episode (configs[4]): cold start, then carried-over scores.
        _case("episode", name="episode", n_3d=1024, steps=8),
        # The same where consecutive frames share most of their content and the program says which rows changed.
        _case("episode", name="episode_reuse", n_3d=1024, steps=8, reuse=True),
        # Eight requests from independent clients, submitted one after another without waiting.
        _case("requests", name="requests_8", requests=8, mode="fixed"),
        # Alg. 1 patch by patch in the paper's host-model shape (256 image patches + 256 point tokens) ...
        _case("patch", name="patch_frame", mode="patch", n_3d=256),
        # ... and batched, with texts of different lengths.
        _case("patch", name="patch_batch_16", mode="patch", batch=16, txt_lo=16, txt_hi=64, n_3d=256),
        # A rank of a four-way head-sharded server: 8 of the 32 heads, replicated hidden rows, four requests.
        _case("shard", name="shard_quarter", batch=4, heads=8, txt_lo=16, txt_hi=48),
    ]


def _log(rng, lo, hi):
    """A whole number between lo and hi, even over its logarithm."""
    return int(round(lo * (hi / lo) ** rng.random()))


def _model(rng):
    return rng.choice([_7B, _7B, {"d_model": 2048, "heads": 16, "head_dim": 128}, {"d_model": 2048, "heads": 32, "head_dim": 64},
                       {"d_model": 3072, "heads": 32, "head_dim": 96}, {"d_model": 4096, "heads": 16, "head_dim": 256}])


def draw(rng):
    c = _draw(rng)
    most = max(work(x)["bytes"] for x in listed())
    while work(c)["bytes"] > most:             # no drawn case costs more than the largest listed one
        c["batch"] -= 1
    return c


def _draw(rng):
    kind = rng.choice(["tiny", "frame", "frame", "batch", "batch", "views", "episode", "requests", "patch", "patch", "shard"])
    lo = rng.randint(4, 48)
    keep = round(rng.uniform(0.15, 0.6), 3)
    c = {"shape": rng.randrange(1 << 20), "txt_lo": lo, "txt_hi": rng.randint(lo, 64), "keep_lo": keep,
         "keep_hi": round(min(0.8, keep + rng.uniform(0.0, 0.3)), 3), "text_first": rng.random() < 0.3}
    if kind == "tiny":
        c.update(rng.choice([{"d_model": 512, "heads": 8, "head_dim": 64}, {"d_model": 1024, "heads": 16, "head_dim": 64},
                             {"d_model": 1024, "heads": 8, "head_dim": 128}]))
        return _case("frame", dtype=rng.choice(["fp32", "fp32", "bf16"]), n_2d=_log(rng, 32, 400), n_3d=_log(rng, 32, 600),
                     mode=rng.choice(["fixed", "adaptive"]), **c)
    if kind == "frame":
        c.update(_model(rng))
        dtype = rng.choice(["bf16", "bf16", "fp8"])
        return _case("frame", dtype=dtype, kv_heads=rng.choice([0, c["heads"] // 4]), n_2d=_log(rng, 64, 800),
                     n_3d=_log(rng, 96, 1200), mode=rng.choice(["fixed", "adaptive"]), **c)
    if kind == "batch":
        c.update(_model(rng))
        return _case("batch", dtype=rng.choice(["bf16", "bf16", "fp8"]), batch=_log(rng, 2, 32),
                     kv_heads=rng.choice([0, 0, c["heads"] // 4]), n_2d=_log(rng, 64, 300), n_3d=_log(rng, 64, 512),
                     mode=rng.choice(["fixed", "adaptive", "adaptive"]), **c)
    if kind == "views":                        # many cameras, a large cloud: up to the most tokens a sample can have
        return _case("batch", batch=rng.randint(1, 7), n_2d=rng.randint(700, 2048), n_3d=rng.randint(800, 2048), **c)
    if kind == "episode":
        c.update(rng.choice([_7B, {"d_model": 2048, "heads": 16, "head_dim": 128}]))
        return _case("episode", n_2d=_log(rng, 100, 400), n_3d=_log(rng, 200, 1200), steps=rng.randint(3, 8),
                     reuse=rng.random() < 0.5, **c)
    if kind == "requests":
        c.update(_model(rng))
        return _case("requests", requests=rng.randint(4, 10), n_2d=_log(rng, 64, 400), n_3d=_log(rng, 96, 800),
                     mode=rng.choice(["fixed", "adaptive"]), **c)
    if kind == "patch":
        p = _log(rng, 48, 600)
        c.update(rng.choice([_7B, {"d_model": 2048, "heads": 16, "head_dim": 128}]))
        return _case("patch", mode="patch", batch=rng.choice([1, 1, _log(rng, 2, 16)]), n_2d=p, n_3d=p, **c)
    ranks = rng.choice([2, 4, 8])
    return _case("shard", batch=_log(rng, 1, 8), n_2d=_log(rng, 64, 400), n_3d=_log(rng, 96, 800),
                 **{**c, "heads": _7B["heads"] // ranks})


# ---------------------------------------------------------------------------------------------- sizes of a case
def _samples(case):
    """The requests of a case, packed back to back; text lengths and keep ratios come from its ``shape``."""
    rng = random.Random(case["shape"])
    out, off = [], 0
    for b in range(case["batch"]):
        n_txt, n2, n3 = rng.randint(case["txt_lo"], case["txt_hi"]), case["n_2d"], case["n_3d"]
        kw = dict(keep_2d=case["keep_2d"], keep_3d=case["keep_3d"], state_slot=b,
                  keep_total=round(rng.uniform(case["keep_lo"], case["keep_hi"]), 3))
        if case["text_first"]:
            s = Sample(seq_off=off, off_txt=0, n_txt=n_txt, off_2d=n_txt, n_2d=n2, off_3d=n_txt + n2, n_3d=n3, **kw)
        else:
            s = layout_2d_3d_txt(off, n_txt, n2, n3, **kw)
        out.append(s)
        off += s.seq_len
    return out


def _kept(case, s, step):
    """Rows that survive (the patch-by-patch rules decide theirs from the data: about a fifth of the visual tokens)."""
    if case["mode"] == "patch":
        return s.n_txt + s.n_vis // 5
    if case["kind"] == "episode" and step == 0:
        return s.n_txt + s.n_vis
    if case["mode"] == "fixed":
        return s.n_txt + int(s.keep_2d * s.n_2d + 0.5) + int(s.keep_3d * s.n_3d + 0.5)
    return s.n_txt + int(s.keep_total * s.n_vis + 0.5)


def work(case):
    e_h = 4 if case["dtype"] == "fp32" else 2
    e_q = 1 if case["dtype"] == "fp8" else e_h
    hd = case["heads"] * case["head_dim"]
    hkv = (case["kv_heads"] or case["heads"]) * case["head_dim"]
    total = {"bytes": 0, "flops": 0}
    for s in _samples(case):
        for step in range(case["steps"]):
            kept = _kept(case, s, step)
            n = s.n_vis * hkv * e_q + s.n_txt * hd * e_q                     # the keys and the text queries
            if case["mode"] != "fixed":
                n += s.n_vis * case["d_model"] * e_h                          # hidden rows, for the feature norms
            n += 2 * kept * (case["d_model"] * e_h + 2 * hkv * e_q)           # surviving rows, read and written
            total["bytes"] += (n + 4 * kept) * case["requests"]
            total["flops"] += 2 * s.n_txt * s.n_vis * hd * case["requests"]
    return total


def tolerance(case):
    # Scores are sums of 32-bit products: 1e-5.  Rows are copies.  Positions and counts are whole: a token on a near-tie
    # of its score with the last kept one may fall either way.
    return {"rel": 1e-5, "max": 1e-3, "differ": 0.005}


# ---------------------------------------------------------------------------------------------- inputs
_DTYPES = {"bf16": torch.bfloat16, "fp32": torch.float32, "fp8": torch.float8_e4m3fn}
_MODES = {"fixed": mvla.MODE_FIXED, "adaptive": mvla.MODE_ADAPTIVE, "patch": mvla.MODE_PATCH}


class _Inputs:
    """Hidden rows of a packed batch and their projections, step by step."""

    def __init__(self, case, samples, gen, rng):
        self.case, self.gen, self.rng, self.samples = case, gen, rng, samples
        self.rows = sum(s.seq_len for s in samples)
        d_model, kv = case["d_model"], case["kv_heads"] or case["heads"]
        self.shapes = [(case["heads"], case["head_dim"]), (kv, case["head_dim"]), (kv, case["head_dim"])]
        self.hidden = self._normal(self.rows, d_model)
        self.w = [self._normal(d_model, h * d) * d_model ** -0.5 for h, d in self.shapes]
        gain = torch.ones(self.rows)
        for s in samples:
            self._salient(s, gain)
        self.hidden *= gain.cuda()[:, None]

    def _normal(self, *shape):
        return torch.randn(*shape, generator=self.gen, device="cuda")

    def _salient(self, s, gain):
        """Scale the salient rows: 5 % spikes; patch by patch: object, robot and unbalanced patches."""
        o2, o3 = s.seq_off + s.off_2d, s.seq_off + s.off_3d
        if self.case["mode"] != "patch":
            for off, n in ((o2, s.n_2d), (o3, s.n_3d)):
                gain[[off + j for j in self.rng.sample(range(n), int(0.05 * n + 0.5))]] = 4.0
            return
        order = self.rng.sample(range(s.n_2d), s.n_2d)
        n_obj, n_rob = max(1, round(0.04 * s.n_2d)), max(1, round(0.12 * s.n_2d))
        for rows, g in ((order[:n_obj], 4.0), (order[n_obj:n_obj + n_rob], 2.0)):
            gain[[o2 + p for p in rows]] = g
            gain[[o3 + p for p in rows]] = g
        rest, fifth = order[1:], s.n_2d // 5
        self.rng.shuffle(rest)
        for rows, g in ((order[:1], 0.05), (rest[:fifth], 0.4), (rest[fifth:2 * fifth], 2.5)):
            gain[[o3 + p for p in rows]] *= g

    def drift(self):
        """The next frame: a tenth of the rows moves by N(0, 0.1); with ``reuse`` one run of visual rows.  Returns the
        program's knowledge of what changed, a byte per row."""
        n = max(1, self.rows // 10)
        if self.case["reuse"]:
            s = self.samples[0]
            first = min(s.off_2d, s.off_3d) + self.rng.randrange(s.n_vis - n + 1)
            rows = list(range(first, first + n))
        else:
            rows = self.rng.sample(range(self.rows), n)
        self.hidden[rows] += 0.1 * self._normal(n, self.case["d_model"])
        mask = torch.zeros(self.rows, dtype=torch.uint8)
        mask[rows] = 1
        return mask.numpy()

    def tensors(self):
        dt = _DTYPES[self.case["dtype"]]
        q, k, v = [(self.hidden @ w).to(dt).view(self.rows, *shape) for w, shape in zip(self.w, self.shapes)]
        return q, k, v, self.hidden.to(torch.float32 if dt == torch.float32 else torch.bfloat16)


def _outputs(ctx, samples, scores=False):
    out = ctx.alloc_outputs(samples, extras=False)
    if scores:
        out.ahat = torch.zeros(sum(s.n_vis for s in samples), dtype=torch.float32, device="cuda")
    for t in (out.out_hidden, out.out_k, out.out_v, out.kept_idx, out.out_offsets, out.budgets):
        t.view(torch.uint8).zero_()
    return out


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    rng = random.Random(seed)
    samples = _samples(case)
    kind, n_req = case["kind"], case["requests"]
    ctx = mvla.PruneContext(dtype=_DTYPES[case["dtype"]], n_heads=case["heads"], head_dim=case["head_dim"], d_model=case["d_model"],
                            max_batch=case["batch"], max_text=64, max_2d=case["n_2d"], max_3d=case["n_3d"],
                            n_state_slots=max(n_req, case["batch"]), tau_2d=0.35, tau_3d=0.65,
                            cold_start_full_keep=int(kind == "episode"), patch_path=int(case["mode"] == "patch"),
                            n_kv_heads=case["kv_heads"], logit_cache=int(case["reuse"]))
    inputs = _Inputs(case, samples, gen, rng)
    state = {"kind": kind, "ctx": ctx, "mode": _MODES[case["mode"]], "samples": samples, "desc": mvla.c_samples(samples), "calls": []}
    if kind == "requests":
        for r in range(n_req):
            one = mvla.c_samples([Sample(**{**vars(s), "state_slot": r}) for s in samples])
            state["calls"].append((one, inputs.tensors(), _outputs(ctx, samples), None))
            inputs.drift()
    else:
        changed = None
        for step in range(case["steps"]):
            if step:
                changed = inputs.drift()
            state["calls"].append((state["desc"], inputs.tensors(), _outputs(ctx, samples, kind == "episode"), changed))
    if case["mode"] == "patch":
        state["u"] = torch.rand(case["batch"] * case["n_2d"], generator=gen, device="cuda")
    state["reuse"] = case["reuse"]
    return state


# ---------------------------------------------------------------------------------------------- the calls
def run(state):
    ctx, mode, kind = state["ctx"], state["mode"], state["kind"]
    desc, (q, k, v, hidden), out, _ = state["calls"][0]
    if kind == "frame":
        ctx.prune_step(0, desc, mode, q, k, v, hidden, flags=mvla.FLAG_RESET_STATE, out=out)
    elif kind == "batch":
        ctx.prune_step(0, state["samples"], mode, q, k, v, hidden, flags=mvla.FLAG_RESET_STATE, out=out)
    elif kind == "patch":
        ctx.prune_step(0, desc, mode, q, k, v, hidden, flags=mvla.FLAG_RESET_STATE, out=out, rand_u=state["u"])
    elif kind == "shard":
        tensor_parallel.prune_step_head_sharded(ctx, 0, state["samples"], mode, q, k, v, hidden, flags=mvla.FLAG_RESET_STATE,
                                                out=out)
        return out.kept_idx, out.out_offsets, out.budgets, out.out_hidden, out.out_k, out.out_v, out.attn
    elif kind == "requests":
        flags = mvla.FLAG_RESET_STATE | mvla.FLAG_INPUTS_STABLE
        for desc, (q, k, v, hidden), out, _ in state["calls"]:
            ctx.prune_step(0, desc, mode, q, k, v, hidden, flags=flags, out=out)
    else:
        flags = mvla.FLAG_RESET_STATE
        for desc, (q, k, v, hidden), out, changed in state["calls"]:
            ctx.prune_step(0, desc, mode, q, k, v, hidden, flags=flags, out=out, changed_rows=changed if state["reuse"] else None)
            flags = 0
    return [(c[2].kept_idx, c[2].out_offsets, c[2].budgets, c[2].out_hidden, c[2].out_k, c[2].out_v) +
            ((c[2].ahat,) if c[2].ahat is not None else ()) for c in state["calls"]]
