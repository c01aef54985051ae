"""Host control flow of the region-aware sampler (Algorithm 1 of the paper) over the C-ABI calls.

The loop owns the latent state and sequences library calls; it performs no arithmetic itself.
What it needs from outside is the velocity model (the DiT of the paper, a stand-in in tests):

    model.full(x, t, store)            -> v            velocity of all N image tokens at time t
                                                        (``store`` = this step refreshes the RIKV cache)
    model.region(x_e, t, edit_idx, n_edit) -> v_e      velocity of the edited tokens only

Both take and return bf16 CUDA tensors.  Everything else is a library call: the Euler update of a
full step and of a region step (``velocity_decay``), the partition after the stabilization steps,
the gather of X^E, the AVDCache criterion (``avd_step``, host scalar), the decayed cached velocity,
and the merge with the one-step-predicted unedited tokens at the end of every run of region steps.

Schedule (``kinds``): one character per sampling step, 'F' = full step, 'R' = region step, in the
order the sampler takes them (time decreasing).  ``paper_schedule`` and ``alternating_schedule``
build the two schedules the tests and the benchmark use.

Requests of one batch need not be at the same step (a request that joined the batch later, or the
conditional / unconditional pair of one guided request, which is simply two batch entries).  With
``offsets`` request b takes its step k at tick ``offsets[b] + k``; at every tick the Euler updates of
all requests share their launches, each request with its own time, step length and decay product,
and a request that has nothing to do in a launch sits it out (NaN scalar, see the header).  The
gather of X^E at the beginning of a run of region steps is made per request on its slice of the batch
when the requests are shifted, the merge at the end too when a hook watches the loop.

When the requests of a tick differ in time the model callbacks receive lists:
    model.full(x, [t_b or None], [store_b])          None = request b is not at a full step
    model.region(x_e, [t_b or None], edit_idx, n_edit)
and must return a value for every batch entry (entries with None are ignored).
"""
from __future__ import annotations

from ctypes import c_float
from dataclasses import dataclass, field

from . import binding


def paper_schedule(T=28, t_st=6, forced=(16,), t_sm=2):
    """Stage schedule of the paper's implementation details, steps indexed T .. 1.

    Stabilization: steps T .. T-t_st+1 full.  Bounds [T-t_st, *forced, t_sm-1]; for consecutive
    (prev, next): region steps prev .. next+2, then one full step at next+1 (cache refresh).  The
    steps below the last bound are full smooth steps.  Returns (kinds, partition_after) where
    partition_after is the number of steps taken before the partition.
    """
    kinds = ["F"] * t_st
    bounds = [T - t_st] + list(forced) + [t_sm - 1]
    for prev, nxt in zip(bounds[:-1], bounds[1:]):
        kinds += ["R"] * (prev - nxt - 1) + ["F"]
    kinds += ["F"] * bounds[-1]
    assert len(kinds) == T, len(kinds)
    return "".join(kinds), t_st


def alternating_schedule(T=28, first_full=6, refresh_every=5, last_full=2):
    """Steps k = 1 .. T: full steps 1 .. first_full, then every ``refresh_every``-th step and the last
    ``last_full`` + 1 steps; the rest are region steps."""
    kinds = []
    for k in range(1, T + 1):
        full = k <= first_full or k > T - last_full - 1 or (k - first_full) % refresh_every == 0
        kinds.append("F" if full else "R")
    return "".join(kinds), first_full


@dataclass
class LoopConfig:
    kinds: str                       # 'F' / 'R' per step
    partition_after: int             # partition runs after this many steps
    timesteps: list                  # t before step k, k = 0 .. T, decreasing; timesteps[T] = end time
    gammas: list                     # timestep-aware decay correction per step
    delta: float                     # AVDCache threshold
    metric: int = binding.METRIC_COSINE
    threshold: float = 0.9


@dataclass
class LoopTrace:
    """What happened, for tests and reports."""
    steps: list = field(default_factory=list)        # request 0: (k, kind, 'full' | 'compute' | 'reuse', scale)
    per_request: list = field(default_factory=list)  # the same list for every request
    model_full_calls: int = 0
    model_region_calls: int = 0
    launches: int = 0


@dataclass
class _Group:
    """Requests with the same offset: they take the same steps at the same ticks."""
    offset: int
    requests: list
    k: int = -1                      # the step taken at the present tick
    partitioned: bool = False
    in_run: bool = False
    t_run: float = 0.0
    product: float = 1.0
    have_cache: bool = False


def _check_rows(got, shape, name, region=False):
    """A velocity of another shape than [B, N, C]: one of all tokens may come without the batch dimension of a single
    request; one of a region step holds its rows at the beginning of each request's, for a single request as many as it
    likes.  Returns how many rows of a request may be read: edited tokens beyond them are reported as
    REGIONE_DEV_BOUNDS and keep their place (only a single request can have fewer than N, so strides stay N)."""
    same = got.numel() == shape[0] * shape[1] * shape[2]
    if not (same or shape[0] == 1 if region else same and shape[max(3 - len(got), 0):] == got):
        raise binding.RegionEError(f"{name} must have shape {shape}, got {tuple(got)}")
    return shape[1] if same else min(shape[1], got.numel() // shape[2])


_NAN = float("nan")
_MAX_RUN = 16                        # sampler steps that one update of X^E applies


class RegionELoop:
    """Buffers and call sequence of one edit (a batch of B independent requests; same schedule,
    optionally shifted against each other by ``offsets``).

    The loop's own work is launch-bound (kernels of 2 to 3 us), so its host side is kept short: addresses
    are looked up once per run (the buffers are the loop's while it runs, ``x`` included), requests that move together share their bookkeeping and
    their calls, a full step's velocity is kept by the Euler update that reads it, and the steps that reuse a
    region step's velocity are applied by that step's update (nothing reads X^E between them)."""

    def __init__(self, B, N, C, cfg: LoopConfig, device="cuda"):
        import torch
        self.B, self.N, self.C, self.cfg = B, N, C, cfg
        i32, bf = torch.int32, torch.bfloat16
        z = lambda *s, dt=bf: torch.zeros(s, dtype=dt, device=device)
        self.mask = z(B, N, dt=torch.uint8)
        self.edit_idx, self.keep_idx, self.slot = z(B, N, dt=i32), z(B, N, dt=i32), z(B, N, dt=i32)
        self.n_edit = z(B, dt=i32)
        self.n_all = torch.full((B,), N, dtype=i32, device=device)
        self.x_e, self.v_cache = z(B, N, C), z(B, N, C)      # capacity N: no host read-back needed
        self.v_last_full = z(B, N, C)
        self.dev_status = z(1, dt=i32)
        self.hook = None             # optional callable(event: str, k: int, tensors: dict)

    def run(self, x, ref, model, stream=None, offsets=None):
        """Runs all steps on ``x`` [B, N, C] bf16 (updated in place); returns (x, trace).

        ``offsets`` [B]: request b takes step k at tick offsets[b] + k (default: all zero)."""
        import torch
        cfg, b, st, hook = self.cfg, binding, self.dev_status, self.hook
        kinds, T, B, N, C = cfg.kinds, len(cfg.kinds), self.B, self.N, self.C
        ts = [float(t) for t in cfg.timesteps[:T + 1]]
        offsets = [0] * B if offsets is None else [int(o) for o in offsets]
        if len(offsets) != B or min(offsets) < 0:
            raise b.RegionEError("offsets must hold one non-negative tick per request")
        if hook is None and min(offsets) == max(offsets):
            return self._run_together(x, ref, model, stream, ts)
        groups = [_Group(o, [r for r in range(B) if offsets[r] == o]) for o in sorted(set(offsets))]
        uniform = len(groups) == 1
        tr = LoopTrace(per_request=[[] for _ in range(B)])

        # ---- the library calls of the loop, over the whole batch (NaN scalar: a request sits a call out) ----
        lib, check, ptr, floats = b.load(), b._check, b._ptr, b._per_request
        bf, shape = torch.bfloat16, (B, N, C)
        p_x, p_xe, p_vl, p_vc = ptr(x, bf, "x"), self.x_e.data_ptr(), self.v_last_full.data_ptr(), self.v_cache.data_ptr()
        p_idx, p_slot, p_ne = self.edit_idx.data_ptr(), self.slot.data_ptr(), self.n_edit.data_ptr()
        p_all, p_st = self.n_all.data_ptr(), st.data_ptr()
        if x.shape != shape:
            raise b.RegionEError(f"x must have shape {shape}, got {tuple(x.shape)}")

        def decay(p_v, scale, dts, p_target, p_keep, p_n, rows=N):
            s = b._stream(stream)                           # (the model may have made another stream current)
            check(lib.regione_velocity_decay(p_v, floats(scale, B, "scale"), floats(dts, B, "dt"), p_target, p_keep, p_n,
                                             B, rows, C, p_st, s), "regione_velocity_decay")
            tr.launches += 1

        def spread(values):
            """(group, value) pairs -> one value per request, NaN for the others; a number when all share it."""
            if uniform:
                return values[0][1]
            out = [_NAN] * B
            for g, val in values:
                for r in g.requests:
                    out[r] = val
            return out

        def listed(value):                                  # (for the hook: always one value per request)
            return value if isinstance(value, list) else [value] * B

        def members(gs):
            return sorted(r for g in gs for r in g.requests)

        one = lambda t_, r: t_[r:r + 1]                     # request r's slice of a batch tensor

        def merge(ending, at_end=False):
            # end of runs of region steps: edited tokens from X^E, unedited tokens by one step of the last full
            # velocity over the whole run (x has not changed since the run began, so it is merged in place)
            if hook is None:
                check(lib.regione_merge(p_x, p_vl, p_xe, p_slot, floats(spread([(g, g.t_run - t) for g, t in ending]), B, "dt"),
                                        B, N, N, C, p_x, p_st, b._stream(stream)), "regione_merge")
                tr.launches += 1
            for g, t in ending:
                g.in_run = False
                for r in g.requests if hook is not None else ():
                    k = T if at_end else g.k
                    hook("merge_in", k, dict(r=r, x=one(x, r), v=one(self.v_last_full, r), x_e=one(self.x_e, r),
                                             slot=one(self.slot, r), dt_unedited=g.t_run - t))
                    b.merge(one(x, r), one(self.v_last_full, r), one(self.x_e, r), one(self.slot, r), g.t_run - t, one(x, r),
                            dev_status=st, stream=stream)
                    hook("merge_out", k, dict(r=r, x=one(x, r)))
                    tr.launches += 1

        def start_runs(starting):
            if uniform:
                check(lib.regione_gather(p_x, p_idx, p_ne, B, N, N, N, 2 * C, p_xe, p_st, b._stream(stream)), "regione_gather")
                tr.launches += 1
            for g in starting:
                g.in_run, g.t_run, g.product, g.have_cache = True, ts[g.k], 1.0, False
                for r in g.requests if not uniform else ():
                    b.gather(one(x, r), one(self.edit_idx, r), one(self.n_edit, r), one(self.x_e, r), dev_status=st,
                             stream=stream)
                    tr.launches += 1

        for tick in range(T + max(offsets)):
            full, region = [], []
            for g in groups:
                k = tick - g.offset
                if 0 <= k < T:
                    g.k = k
                    (full if kinds[k] == "F" else region).append(g)
            k0 = groups[0].k if uniform else tick

            # ---- full steps ----
            if full:
                ending = [(g, ts[g.k]) for g in full if g.in_run]
                if ending:
                    merge(ending)
                if uniform:
                    g = full[0]
                    v = model.full(x, ts[g.k], g.partitioned or g.k + 1 == cfg.partition_after)
                else:
                    t_full, store = [None] * B, [False] * B
                    for g in groups:
                        live = 0 <= tick - g.offset < T
                        for r in g.requests:
                            store[r] = live and (g.partitioned or g.k + 1 == cfg.partition_after)
                            if g in full:
                                t_full[r] = ts[g.k]
                    v = model.full(x, t_full, store)
                tr.model_full_calls += 1
                p_v = ptr(v, bf, "v")
                if v.shape != shape:
                    _check_rows(v.shape, shape, "v")
                dts = spread([(g, ts[g.k] - ts[g.k + 1]) for g in full])
                if hook is not None:
                    hook("euler_in", k0, dict(x=x, v=v, dt=listed(dts), active=members(full)))
                decay(p_v, 1.0, dts, p_x, p_vl, p_all)       # (keeps v as the last full velocity in passing)
                if hook is not None:
                    hook("euler_out", k0, dict(x=x, active=members(full)))
                part = [g for g in full if g.k + 1 == cfg.partition_after]
                if part:
                    t_part = spread([(g, ts[g.k + 1]) for g in part])
                    if hook is not None:
                        hook("partition_in", k0, dict(x=x, v=v, ref=ref, t=listed(t_part), active=members(part)))
                    b.partition(x, v, ref, t_part, cfg.metric, cfg.threshold, self.mask, self.edit_idx,
                                self.keep_idx, self.slot, self.n_edit, dev_status=st, stream=stream)
                    if hook is not None:
                        hook("partition_out", k0, dict(mask=self.mask, edit_idx=self.edit_idx, slot=self.slot,
                                                       n_edit=self.n_edit, active=members(part)))
                    tr.launches += 1
                    for g in part:
                        g.partitioned = True
                for g in full:
                    for r in g.requests:
                        tr.per_request[r].append((g.k, "F", "full", 1.0))

            # ---- region steps ----
            if region:
                starting = [g for g in region if not g.in_run]
                if any(not g.partitioned for g in starting):
                    raise b.RegionEError("a region step was scheduled before the partition")
                if starting:
                    start_runs(starting)
                reuse, compute = [], []
                for g in region:
                    again = False
                    if g.have_cache:
                        g.product, again = b.avd_step(g.product, ts[g.k - 1] - ts[g.k], float(cfg.gammas[g.k]), cfg.delta)
                    (reuse if again else compute).append(g)
                for gs, kind in ((reuse, "reuse"), (compute, "compute")):
                    if not gs:
                        continue
                    scale = spread([(g, g.product if kind == "reuse" else 1.0) for g in gs])
                    dts = spread([(g, ts[g.k] - ts[g.k + 1]) for g in gs])
                    v_e, p_v, p_keep, rows = self.v_cache, p_vc, None, N
                    if kind == "compute":
                        if uniform:
                            v_e = model.region(self.x_e, ts[gs[0].k], self.edit_idx, self.n_edit)
                        else:
                            t_e = [None] * B
                            for g in gs:
                                for r in g.requests:
                                    t_e[r] = ts[g.k]
                            v_e = model.region(self.x_e, t_e, self.edit_idx, self.n_edit)
                        tr.model_region_calls += 1
                        p_v, p_keep = ptr(v_e, bf, "v_e"), p_vc
                        if v_e.shape != shape:
                            rows = _check_rows(v_e.shape, shape, "v_e", region=True)
                    if hook is not None:
                        hook("decay_in", k0, dict(v=v_e, x_e=self.x_e, scale=listed(scale), dt=listed(dts),
                                                  n_edit=self.n_edit, active=members(gs)))
                    decay(p_v, scale, dts, p_xe, p_keep, p_ne, rows)
                    if hook is not None:
                        hook("decay_out", k0, dict(x_e=self.x_e, active=members(gs)))
                    for g in gs:
                        if kind == "compute":
                            g.product, g.have_cache = 1.0, True
                        for r in g.requests:
                            tr.per_request[r].append((g.k, "R", kind, g.product))

            # requests whose last step was a region step end with the merge
            ending = [(g, ts[T]) for g in region if g.k == T - 1]
            if ending:
                merge(ending, at_end=True)
        tr.steps = tr.per_request[0]
        return x, tr

    def _run_together(self, x, ref, model, stream, ts):
        """All steps of requests that take them at the same time, without a hook: what ``run`` does then, with one
        set of scalars for the batch.  Host-bound (28 steps of 4096 tokens, 12 of them full: about 6 us a launch, 237 us
        with a launch for each of the loop's operations, 203 us this way), so an update and what the loop does next to
        the same rows are one call: a full step and the gather of X^E behind it, the last update of a run of region
        steps and the merge.  Not where the velocity lies in the rows that the second half writes (a model may return
        its latent, or a buffer of the loop): other blocks may not have read it yet."""
        import torch
        cfg, b = self.cfg, binding
        kinds, after, gammas, delta = cfg.kinds, cfg.partition_after, cfg.gammas, cfg.delta
        T, B, N, C = len(kinds), self.B, self.N, self.C
        lib, check, ptr, avd_step = b.load(), b._check, b._ptr, b.avd_step
        bf, shape, s = torch.bfloat16, (B, N, C), b._stream(stream)
        # (the model may make another stream current: looked up again behind each of its calls)
        follow, stream_of, device = stream is None, torch._C._cuda_getCurrentRawStream, torch._C._cuda_getDevice
        p_x, p_xe, p_vl, p_vc = ptr(x, bf, "x"), self.x_e.data_ptr(), self.v_last_full.data_ptr(), self.v_cache.data_ptr()
        p_slot, p_ne, p_st = (t.data_ptr() for t in (self.slot, self.n_edit, self.dev_status))
        if x.shape != shape:
            raise b.RegionEError(f"x must have shape {shape}, got {tuple(x.shape)}")
        plan = b.LoopPlan(B, N, C, p_x, p_xe, p_vl, p_vc, p_slot, p_ne, p_st)
        one, full_step, region_steps = c_float * B, lib.regione_loop_full_step, lib.regione_loop_region_steps
        n_bytes = 2 * B * N * C
        log, launches, full_calls, region_calls = [], 0, 0, 0
        partitioned, t_run, k = False, None, 0               # t_run: time at which the present run of region steps began

        while k < T or t_run is not None:
            if t_run is not None and (k == T or kinds[k] == "F"):     # (not part of the last update: see above)
                # x has not changed since the run began: edited tokens from X^E, the others by one step of the last
                # full velocity over the whole run
                check(lib.regione_merge(p_x, p_vl, p_xe, p_slot, one(*[t_run - ts[k]] * B), B, N, N, C, p_x, p_st, s),
                      "regione_merge")
                launches += 1
                t_run = None
                if k == T:
                    break
            if kinds[k] == "F":
                t, t_next = ts[k], ts[k + 1]
                last_before = k + 1 == after
                v = model.full(x, t, partitioned or last_before)
                if follow:
                    s = stream_of(device())
                full_calls += 1
                p_v = ptr(v, bf, "v")
                if v.shape != shape:
                    _check_rows(v.shape, shape, "v")
                starts = partitioned and k + 1 < T and kinds[k + 1] == "R" and abs(p_v - p_xe) >= n_bytes
                check(full_step(plan, p_v, one(*[t - t_next] * B), starts, s), "regione_loop_full_step")
                launches += 1
                if starts:
                    t_run = t_next
                if last_before:
                    b.partition(x, v, ref, t_next, cfg.metric, cfg.threshold, self.mask, self.edit_idx, self.keep_idx,
                                self.slot, self.n_edit, dev_status=self.dev_status, stream=stream)
                    launches += 1
                    partitioned = True
                log.append((k, "F", "full", 1.0))
                k += 1
                continue
            if t_run is None:
                if not partitioned:
                    raise b.RegionEError("a region step was scheduled before the partition")
                check(lib.regione_gather(p_x, self.edit_idx.data_ptr(), p_ne, B, N, N, N, 2 * C, p_xe, p_st, s),
                      "regione_gather")
                launches += 1
                t_run = ts[k]
            v_e = model.region(self.x_e, ts[k], self.edit_idx, self.n_edit)
            if follow:
                s = stream_of(device())
            region_calls += 1
            p_v, rows = ptr(v_e, bf, "v_e"), N
            if v_e.shape != shape:
                rows = _check_rows(v_e.shape, shape, "v_e", region=True)
            log.append((k, "R", "compute", 1.0))
            scales, dts, product, again = [1.0] * B, [ts[k] - ts[k + 1]] * B, 1.0, True
            first, k = k, k + 1
            while again:
                again = False
                if k < T and kinds[k] == "R":
                    product, again = avd_step(product, ts[k - 1] - ts[k], float(gammas[k]), delta)
                if again and k - first < _MAX_RUN:
                    log.append((k, "R", "reuse", product))
                    scales += [product] * B
                    dts += [ts[k] - ts[k + 1]] * B
                    k += 1
                    continue
                # (a run that is longer than one update carries goes on in the next, from the kept velocity)
                n = k - first
                many = c_float * (n * B)
                if rows == N:
                    ends = not again and (k == T or kinds[k] == "F") and (p_v is None or abs(p_v - p_x) >= n_bytes)
                    check(region_steps(plan, p_v, many(*scales), many(*dts), n, one(*[t_run - ts[k]] * B) if ends else None, s),
                          "regione_loop_region_steps")
                    if ends:
                        t_run = None
                else:
                    check(lib.regione_velocity_decay_run(p_v, many(*scales), many(*dts), n, p_xe, p_vc, p_ne, B, rows, C, p_st, s),
                          "regione_velocity_decay_run")
                launches += 1
                if again:
                    log.append((k, "R", "reuse", product))
                    p_v, rows, first, scales, dts = None, N, k, [product] * B, [ts[k] - ts[k + 1]] * B
                    k += 1
        return x, LoopTrace(log, [list(log) for _ in range(B)], full_calls, region_calls, launches)
