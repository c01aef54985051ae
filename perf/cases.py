"""The work that a user of this package has it do, as cases that can be timed and compared.

Every case is a dict of plain values; ``kind`` names the part of the sampler it stands for:

  step       one region-aware denoising step of one attention layer (``RegionStep.run``), either refreshing
             the Region-Instruction KV cache from the step's own K / V or attending over the cache an
             earlier step left
  full       the attention of a full step over the joint sequence, plain (stabilization and smoothing
             steps) or refreshing the cache in the same call (the step before a run of region steps)
  layer      a region step's attention layer as a transformer block calls it: rows projected compactly,
             normalised and rotated at their own positions, then attention over [fresh | cached]
  quant      the 8-bit cache: encoding a layer's retained rows, or decoding them and attending over them
  loop       the 28-step sampler of one batch of edits around a given velocity (latent updates, partition,
             criterion and merges; the model's own time is not in it)

``listed`` holds the shapes the configurations of this repository name; ``draw`` gives more of the same
ranges.  Q and K are drawn so that the logits have unit variance (what normalised queries and keys give),
latents follow the flow-matching construction with a planted region (see ``_latents``).
"""
import math

import torch

from paper_2510_25590_b200 import binding, synth
from paper_2510_25590_b200.loop import LoopConfig, RegionELoop, alternating_schedule, paper_schedule
from paper_2510_25590_b200.step import RegionStep, StepShapes

C = 16                            # latent channels of every configuration
THRESHOLD = {"cosine": 0.88, "l2": 0.1}
METRIC = {"cosine": binding.METRIC_COSINE, "l2": binding.METRIC_L2}
MEMBERSHIP = {"edited": binding.ROWS_EDITED_QUERIES, "paper": binding.ROWS_PAPER}
T_PARTITION = 22.0 / 28.0         # time at which the partition runs: after 6 of 28 steps
MOST_FLOPS = 1.2e12               # a drawn case costs no more than the largest listed one


def listed():
    flux = dict(B=1, rows=64, cols=64, n_ref=4096, n_text=512, H=24, D=128)       # 1024 x 1024 image
    qwen = dict(B=1, rows=64, cols=64, n_ref=4096, n_text=256, H=24, D=128)
    large = dict(B=4, rows=96, cols=96, n_ref=9216, n_text=512, H=24, D=128)      # four 1536 x 1536 edits in one batch
    cos = dict(metric="cosine", members="edited")
    return [
        # a thumbnail-sized edit: launches and host time
        dict(name="step_tiny_store", kind="step", B=1, rows=32, cols=32, n_ref=1024, n_text=64, H=4, D=64,
             ratio=0.25, store=True, **cos),
        # the benchmark's workload: a fifth of the image edited, cache taken from this step's K / V
        dict(name="step_flux_store", kind="step", ratio=0.20, store=True, **flux, **cos),
        # the same layer in the region steps that follow, which only read the cache
        dict(name="step_flux_reuse", kind="step", ratio=0.20, store=False, **flux, **cos),
        # a small retouch: 205 queries (a ragged second tile) against the whole context
        dict(name="step_qwen_5pct_reuse", kind="step", ratio=0.05, store=False, **qwen, **cos),
        # a large edit
        dict(name="step_qwen_50pct_store", kind="step", ratio=0.50, store=True, **qwen, **cos),
        # four high-resolution requests, each with its own mask, in one launch
        dict(name="step_large_batch4_store", kind="step", ratio=0.15, store=True, **large, **cos),
        # full step that leaves the cache for the region steps behind it
        dict(name="full_qwen_store", kind="full", ratio=0.20, store=True, **qwen),
        # full step of the stabilization stage
        dict(name="full_flux", kind="full", ratio=0.20, store=False, **flux),
        # one block's attention in a region step, text rows recomputed as the paper's equation has it
        dict(name="layer_step1x_paper", kind="layer", ratio=0.20, rope="interleaved", **qwen),
        # region step on the 8-bit cache: decode and attend
        dict(name="quant_flux_decode", kind="quant", encode=False, ratio=0.20, **flux),
        # full step of four high-resolution requests: encode one layer's retained rows
        dict(name="quant_large_encode", kind="quant", encode=True, ratio=0.15, **large),
        # the sampler's own work over 28 steps of one 1024 x 1024 edit
        dict(name="loop_step1x_28", kind="loop", B=1, rows=64, cols=64, ratio=0.20, metric="l2", paper=False,
             shift=0),
    ]


def draw(rng):
    def near(lo, hi):                                   # log-uniform whole number
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["step", "step", "step", "step", "full", "full", "layer", "quant", "loop"])
    for _ in range(1000):
        c = dict(kind=kind, B=rng.choice([1, 1, 1, 2, 3, 4]), rows=near(24, 96), cols=near(24, 96),
                 ratio=round(math.exp(rng.uniform(math.log(0.03), math.log(1.0))), 3))
        if kind in ("step", "full", "layer", "quant"):
            img = c["rows"] * c["cols"]
            c.update(n_ref=img if rng.random() < 0.7 else near(500, 9216), n_text=near(20, 512),
                     H=rng.choice([4, 8, 12, 16, 24, 24, 24]), D=rng.choice([64, 128, 128, 128]))
        if kind == "step":
            c.update(metric=rng.choice(["cosine", "cosine", "l2"]), members=rng.choice(["edited", "edited", "paper"]),
                     store=rng.random() < 0.5)
        elif kind == "full":
            c.update(store=rng.random() < 0.5)
        elif kind == "layer":
            c.update(rope=rng.choice(["interleaved", "half"]))
        elif kind == "quant":
            c.update(encode=rng.random() < 0.5)
        else:
            c.update(metric=rng.choice(["cosine", "l2"]), paper=rng.random() < 0.5, shift=rng.choice([0, 0, 3]))
        w = work(c)
        if w["flops"] <= MOST_FLOPS and w["bytes"] <= 1.2e9:
            return c
    raise AssertionError("no case of the range found")


# ------------------------------------------------------------------------------------------------
# counts
# ------------------------------------------------------------------------------------------------


def _counts(case):
    """Image tokens, edited tokens, and rows of the joint sequence of one request."""
    n_img = case["rows"] * case["cols"]
    return n_img, max(1, int(round(case["ratio"] * n_img))), case.get("n_text", 0) + n_img + case.get("n_ref", 0)


def _region_counts(case, paper):
    n_img, n_edit, n_full = _counts(case)
    n_q = n_edit + (case["n_text"] if paper else 0)
    return n_q, n_full - n_q


def work(case):
    """Bytes and operations of one pass that no implementation can do without (per request times B)."""
    B, kind = case["B"], case["kind"]
    n_img, n_edit, n_full = _counts(case)
    row = case.get("H", 0) * case.get("D", 0) * 2                    # one token's K (or Q, V, O) of all heads
    lat = C * 2
    search = n_img * (3 * lat + 1 + 4 + 4)                           # three latents in; mask, slot, list out
    if kind == "loop":
        ts = 28
        return dict(bytes=B * (ts * n_edit * 3 * lat + 12 * (n_img - n_edit) * 3 * lat + search), flops=0)
    paper = kind == "layer" or case.get("members") == "paper"
    n_q, n_c = _region_counts(case, paper)
    flops = 4.0 * case["H"] * case["D"] * n_q * n_full
    if kind == "full":
        keep = (n_full - n_edit) if case["store"] else 0
        return dict(bytes=B * (4 * n_full + 2 * keep) * row, flops=B * 4.0 * case["H"] * case["D"] * n_full * n_full)
    if kind == "step":
        move = search + 4 * n_full + 2 * n_img * lat + 2 * n_edit * lat             # partition, lists, update and merge
        move += (2 * n_q + 2 * n_full) * row                                        # Q in, O out, every K and V row in
        move += 2 * n_c * row if case["store"] else 0                               # cache out
        return dict(bytes=B * move, flops=B * flops)
    if kind == "layer":
        return dict(bytes=B * ((3 + 3 + 1) * n_q + 2 * n_c) * row, flops=B * flops)  # Q, K, V in and out, O out
    quant = n_c * case["H"] * (2 * case["D"] + 8)                                   # codes and scales of K and V
    if case["encode"]:
        return dict(bytes=B * (2 * n_c * row + quant), flops=0)
    return dict(bytes=B * (quant + 2 * n_c * row + 4 * n_q * row), flops=B * flops)  # widened cache is a result too


def tolerance(case):
    if case.get("encode"):
        return "exact"                        # codes and power-of-two scales
    # bf16 results of an attention whose probabilities are rounded to bf16 before the second product: against the
    # same attention in 64 bits every listed case shows rel 2.2e-3 to 2.4e-3 and at most 1.4e-2 of the result's scale
    return dict(rel=1e-2, max=6e-2)


# ------------------------------------------------------------------------------------------------
# inputs
# ------------------------------------------------------------------------------------------------


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _randn(g, *shape, std=1.0):
    x = torch.randn(shape, generator=g, device="cuda", dtype=torch.bfloat16)
    return x if std == 1.0 else x * std


def _masks(g, case):
    """Planted edit masks [B, N]: smooth random fields cut at the level that edits exactly ``ratio``."""
    B, rows, cols = case["B"], case["rows"], case["cols"]
    n_img, n_edit, _ = _counts(case)
    y = torch.arange(rows, device="cuda", dtype=torch.float32)[:, None] / max(rows, cols)
    x = torch.arange(cols, device="cuda", dtype=torch.float32)[None, :] / max(rows, cols)
    p = torch.rand((B, 8, 3, 1, 1), generator=g, device="cuda")
    f = torch.sin(2 * math.pi * ((6 * p[:, :, 0] - 3) * y + (6 * p[:, :, 1] - 3) * x + p[:, :, 2])).sum(1)
    f = f.reshape(B, n_img) + 1e-4 * torch.rand((B, n_img), generator=g, device="cuda")
    m = torch.zeros((B, n_img), dtype=torch.bool, device="cuda")
    return m.scatter_(1, f.topk(n_edit, dim=1).indices, True)


def _latents(g, case, t=T_PARTITION):
    """x_t, v, ref [B, N, 16]: outside the planted region the clean target is the reference latent up to a
    small perturbation, inside it is unrelated to it; v is the straight-line velocity."""
    m = _masks(g, case)[:, :, None]
    n = (case["B"], case["rows"] * case["cols"], C)
    r, noise, z, small = (torch.randn(n, generator=g, device="cuda") for _ in range(4))
    r = r.bfloat16().float()
    x0 = torch.where(m, math.sqrt(0.91) * z - 0.3 * r, r + 0.005 * small)
    v = noise - x0
    return ((1.0 - t) * x0 + t * noise).bfloat16(), v.bfloat16(), r.bfloat16(), m[:, :, 0]


def _i32(*shape):
    return torch.zeros(shape, dtype=torch.int32, device="cuda")


def _full_i32(B, value):
    return torch.full((B,), value, dtype=torch.int32, device="cuda")


def _workspace(n_bytes):
    return torch.empty(max(int(n_bytes), 256), dtype=torch.uint8, device="cuda")


def _row_lists(g, case, paper):
    """Recomputed and cached rows of the joint sequence, [B, n_q] and [B, n_c] int32, ascending."""
    n_text, n_img = case["n_text"], case["rows"] * case["cols"]
    n_q, n_c = _region_counts(case, paper)
    live = torch.zeros((case["B"], _counts(case)[2]), dtype=torch.bool, device="cuda")
    live[:, n_text:n_text + n_img] = _masks(g, case)
    live[:, :n_text] = paper
    rows = lambda m, n: m.nonzero()[:, 1].view(case["B"], n).int().contiguous()
    return rows(live, n_q), rows(~live, n_c)


def prepare(case, seed):
    return {"step": _prepare_step, "full": _prepare_full, "layer": _prepare_layer, "quant": _prepare_quant,
            "loop": _prepare_loop}[case["kind"]](case, _gen(seed))


def run(state):
    return state["run"](state)


# ---- one region-aware step -------------------------------------------------------------------------


def _prepare_step(case, g):
    x_t, v, ref, _ = _latents(g, case)
    B, H, D = case["B"], case["H"], case["D"]
    n_img, n_edit, n_full = _counts(case)
    qkv = [_randn(g, B, n_full, H, D) for _ in range(3)]
    cap = (n_edit + 127) // 128 * 128                  # what plan_capacity returns for these latents
    step = RegionStep(StepShapes(B, n_img, case["n_text"], case["n_ref"], C, H, D, cap, METRIC[case["metric"]],
                                 THRESHOLD[case["metric"]], MEMBERSHIP[case["members"]]))
    if not case["store"]:                              # the cache that an earlier step left: other K and V
        step.k_cache.copy_(_randn(g, B, n_full, H, D))
        step.v_cache.copy_(_randn(g, B, n_full, H, D))
    return dict(run=_run_step, step=step, args=(x_t, v, ref, *qkv, T_PARTITION, 0.97, 1.0 / 28.0, 5.0 / 28.0),
                store=case["store"])


def _run_step(s):
    step = s["step"]
    step.run(*s["args"], store_cache=s["store"])
    out = dict(x_out=step.x_out, o_full=step.o_full, x_e=step.x_e, v_avd=step.v_avd, mask=step.mask, slot=step.slot,
               n_edit=step.n_edit, n_q=step.n_q, n_cache=step.n_cache, query_rows=step.query_rows,
               cache_rows=step.cache_rows, status=step.dev_status)
    if s["store"]:
        out.update(k_cache=step.k_cache, v_cache=step.v_cache)
    return out


# ---- attention of a full step ----------------------------------------------------------------------


def _prepare_full(case, g):
    B, H, D = case["B"], case["H"], case["D"]
    n_full = _counts(case)[2]
    q, k, v = (_randn(g, B, n_full, H, D) for _ in range(3))
    s = dict(q=q, k=k, v=v, n=_full_i32(B, n_full), zero=_i32(B), out=torch.zeros_like(q), status=_i32(1))
    if not case["store"]:
        s.update(run=_run_full, workspace=_workspace(binding.region_attention_workspace(B, n_full, n_full, 0, H, D)))
        return s
    _, keep = _row_lists(g, case, False)
    n_c = keep.shape[1]
    s.update(run=_run_full_store, keep=keep, n_keep=_full_i32(B, n_c), k_cache=torch.zeros_like(k[:, :n_c]).contiguous(),
             v_cache=torch.zeros_like(v[:, :n_c]).contiguous(),
             workspace=_workspace(binding.full_attention_store_workspace(B, n_full, H, D)))
    return s


def _run_full(s):
    binding.region_attention(s["q"], s["k"], s["v"], None, None, s["n"], s["n"], s["zero"], s["out"],
                             workspace=s["workspace"], dev_status=s["status"])
    return s["out"], s["status"]


def _run_full_store(s):
    binding.full_attention_store(s["q"], s["k"], s["v"], s["n"], s["keep"], s["n_keep"], s["k_cache"], s["v_cache"],
                                 s["out"], workspace=s["workspace"], dev_status=s["status"])
    return s["out"], s["k_cache"], s["v_cache"], s["status"]


# ---- a block's attention layer in a region step ------------------------------------------------------


def _prepare_layer(case, g):
    B, H, D = case["B"], case["H"], case["D"]
    n_full = _counts(case)[2]
    rows, _ = _row_lists(g, case, True)
    n_q, n_c = _region_counts(case, True)
    cos, sin = (torch.from_numpy(a).cuda() for a in synth.rope_tables(n_full, D))
    new = lambda: torch.zeros((B, n_q, H, D), dtype=torch.bfloat16, device="cuda")
    return dict(run=_run_layer, src=[_randn(g, B, n_q, H, D) for _ in range(3)], rows=rows, n_q=_full_i32(B, n_q),
                n_c=_full_i32(B, n_c), wq=1 + _randn(g, D, std=0.1), wk=1 + _randn(g, D, std=0.1), cos=cos, sin=sin,
                layout=binding.ROPE_HALF if case["rope"] == "half" else binding.ROPE_INTERLEAVED,
                q=new(), k=new(), v=new(), out=new(), k_cache=_randn(g, B, n_c, H, D), v_cache=_randn(g, B, n_c, H, D),
                workspace=_workspace(binding.region_attention_workspace(B, n_q, n_q, n_c, H, D)), status=_i32(1))


def _run_layer(s):
    binding.fresh_qkv(*s["src"], s["rows"], s["n_q"], s["wq"], s["wk"], 1e-6, s["cos"], s["sin"], s["layout"],
                      s["q"], s["k"], s["v"], src_compact=True, dev_status=s["status"])
    binding.region_attention(s["q"], s["k"], s["v"], s["k_cache"], s["v_cache"], s["n_q"], s["n_q"], s["n_c"], s["out"],
                             workspace=s["workspace"], dev_status=s["status"])
    return s["q"], s["k"], s["v"], s["out"], s["status"]


# ---- the 8-bit cache ---------------------------------------------------------------------------------


def _prepare_quant(case, g):
    B, H, D = case["B"], case["H"], case["D"]
    n_full = _counts(case)[2]
    rows, keep = _row_lists(g, case, False)
    n_q, n_c = _region_counts(case, False)
    codes = lambda: torch.zeros((B, n_c, H, D), dtype=torch.uint8, device="cuda")
    scales = lambda: torch.zeros((B, n_c, H), dtype=torch.float32, device="cuda")
    s = dict(k_full=_randn(g, B, n_full, H, D), v_full=_randn(g, B, n_full, H, D), keep=keep, n_c=_full_i32(B, n_c),
             k_q=codes(), v_q=codes(), k_s=scales(), v_s=scales(), status=_i32(1))
    if case["encode"]:
        s.update(run=_run_encode)
        return s
    _run_encode(s)                                      # an earlier full step left the codes
    del s["k_full"], s["v_full"]
    wide = lambda: torch.zeros((B, n_c, H, D), dtype=torch.bfloat16, device="cuda")
    s.update(run=_run_decode, n_q=_full_i32(B, n_q), q=_randn(g, B, n_q, H, D), k=_randn(g, B, n_q, H, D),
             v=_randn(g, B, n_q, H, D), k_cache=wide(), v_cache=wide(),
             out=torch.zeros((B, n_q, H, D), dtype=torch.bfloat16, device="cuda"),
             workspace=_workspace(binding.region_attention_workspace(B, n_q, n_q, n_c, H, D)))
    return s


def _run_encode(s):
    binding.rikv_store_e4m3(s["k_full"], s["v_full"], s["keep"], s["n_c"], s["k_q"], s["v_q"], s["k_s"], s["v_s"],
                            dev_status=s["status"])
    return s["k_q"], s["v_q"], s["k_s"], s["v_s"], s["status"]


def _run_decode(s):
    binding.rikv_load_e4m3(s["k_q"], s["v_q"], s["k_s"], s["v_s"], s["n_c"], s["k_cache"], s["v_cache"],
                           dev_status=s["status"])
    binding.region_attention(s["q"], s["k"], s["v"], s["k_cache"], s["v_cache"], s["n_q"], s["n_q"], s["n_c"], s["out"],
                             workspace=s["workspace"], dev_status=s["status"])
    return s["out"], s["k_cache"], s["v_cache"], s["status"]


# ---- the 28-step sampler -----------------------------------------------------------------------------


class _GivenVelocity:
    """A velocity model that costs nothing of its own: the straight-line velocity of every token, and its
    edited rows for a region step (gathered by the library, as a model would take its rows)."""

    def __init__(self, v, case):
        self.v, self.v_e, self.status = v, torch.zeros_like(v), _i32(1)

    def full(self, x, t, store):
        return self.v

    def region(self, x_e, t, edit_idx, n_edit):
        binding.gather(self.v, edit_idx, n_edit, self.v_e, dev_status=self.status)
        return self.v_e


def _prepare_loop(case, g):
    noise, v, ref, _ = _latents(g, case, t=1.0)         # the sampler starts from noise
    kinds, after = paper_schedule() if case["paper"] else alternating_schedule()
    T = len(kinds)
    cfg = LoopConfig(kinds, after, [1.0 - k / T for k in range(T + 1)], [1.0] * (T + 1), 0.05, METRIC[case["metric"]],
                     THRESHOLD[case["metric"]])
    B, N, _ = noise.shape
    return dict(run=_run_loop, loop=RegionELoop(B, N, C, cfg), model=_GivenVelocity(v, case), noise=noise, ref=ref,
                x=torch.empty_like(noise), offsets=[case["shift"] * b for b in range(B)] if case["shift"] else None)


def _run_loop(s):
    s["x"].copy_(s["noise"])
    x, _ = s["loop"].run(s["x"], s["ref"], s["model"], offsets=s["offsets"])
    lp = s["loop"]
    return dict(x=x, mask=lp.mask, slot=lp.slot, n_edit=lp.n_edit, x_e=lp.x_e, status=lp.dev_status)
