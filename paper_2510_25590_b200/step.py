"""One region-aware denoising step for one attention layer, as one C-ABI call.

This is buffer ownership only (torch tensors are device buffers): every operation runs in the
library's kernels.  The sequence follows Algorithm 1 of the paper for one layer:

  partition with the joint-sequence row lists -> gather X^E, v^E; velocity decay + Euler update; merge with
  the one-step-predicted unedited tokens; gather of the recomputed rows of Q (K, V) -> region attention
  writing its rows back at their joint-sequence positions, the RIKV store in the same launch

(three kernel launches: partition, moves, attention; a fourth where a kernel of its own merges the attention's shared
items.  `regione_kernel_launches` counts them).

No step needs a host round trip: per-request counts stay in device memory.
Capacities are host integers chosen by the caller (``plan_capacity`` reads the
edited-token count back once, outside any timed region).
"""
from __future__ import annotations

from dataclasses import dataclass

from . import binding


@dataclass
class StepShapes:
    B: int
    N: int          # image tokens
    n_text: int
    n_ref: int
    C: int          # latent channels
    H: int
    D: int
    ne_cap: int     # capacity for edited tokens (rows of X^E)
    metric: int = binding.METRIC_COSINE
    threshold: float = 0.9
    membership: int = binding.ROWS_EDITED_QUERIES

    @property
    def n_full(self):
        return self.n_text + self.N + self.n_ref

    @property
    def q_cap(self):
        return self.ne_cap + (self.n_text if self.membership == binding.ROWS_PAPER else 0)

    @property
    def c_cap(self):
        return self.n_full          # the cache can never hold more than the joint sequence


def plan_capacity(x_t, v, ref, t, metric, threshold, round_to=128):
    """Runs the partition once and returns max_b n_edit[b] rounded up (one host read-back)."""
    import torch
    B, N, _ = x_t.shape
    dev = x_t.device
    mask = torch.empty((B, N), dtype=torch.uint8, device=dev)
    e, k, s = (torch.empty((B, N), dtype=torch.int32, device=dev) for _ in range(3))
    ne = torch.empty(B, dtype=torch.int32, device=dev)
    binding.partition(x_t, v, ref, t, metric, threshold, mask, e, k, s, ne)
    m = int(ne.max().item())
    return max(round_to, (m + round_to - 1) // round_to * round_to)


class RegionStep:
    """Owns the intermediate buffers of one step and launches its kernels in order."""

    def __init__(self, shp: StepShapes, device="cuda"):
        import torch
        self.shp = shp
        B, N, C, H, D = shp.B, shp.N, shp.C, shp.H, shp.D
        i32, bf = torch.int32, torch.bfloat16
        z = lambda *s, dt=bf: torch.zeros(s, dtype=dt, device=device)
        self.mask = z(B, N, dt=torch.uint8)
        self.edit_idx, self.keep_idx, self.slot = z(B, N, dt=i32), z(B, N, dt=i32), z(B, N, dt=i32)
        self.n_edit, self.n_q, self.n_cache = z(B, dt=i32), z(B, dt=i32), z(B, dt=i32)
        self.query_rows, self.cache_rows = z(B, shp.q_cap, dt=i32), z(B, shp.c_cap, dt=i32)
        self.x_e, self.v_e, self.v_avd = z(B, shp.ne_cap, C), z(B, shp.ne_cap, C), z(B, shp.ne_cap, C)
        self.k_cache, self.v_cache = z(B, shp.c_cap, H, D), z(B, shp.c_cap, H, D)
        self.q_e, self.k_fresh, self.v_fresh = (z(B, shp.q_cap, H, D) for _ in range(3))
        self.o_e = z(B, shp.q_cap, H, D)
        self.o_full = z(B, shp.n_full, H, D)
        self.x_out = z(B, N, C)
        self.dev_status = z(1, dt=i32)
        self.n_rows = torch.full((B,), shp.n_full, dtype=i32, device=device)
        self.workspace = torch.empty(max(binding.region_step_workspace(self._new_plan()), 256), dtype=torch.uint8,
                                     device=device)
        self.launches = 0                 # operations of the sequence run so far (8 per step, 7 without the store), however
                                          # many kernels they took
        self.kernel_launches = 0          # kernels launched so far, as the library counts them
        self.attention_events = None      # optional (start, stop) pair recorded around the attention
        self._step_plan()

    _BUFFERS = ("mask", "edit_idx", "keep_idx", "slot", "n_edit", "query_rows", "n_q", "cache_rows", "n_cache", "n_rows",
                "x_e", "v_e", "v_avd", "x_out", "q_e", "k_fresh", "v_fresh", "k_cache", "v_cache", "o_full", "workspace",
                "dev_status")

    def __setattr__(self, name, value):
        object.__setattr__(self, name, value)
        if name in self._BUFFERS or name == "shp":
            object.__setattr__(self, "_plan_of", None)   # the plan names this object's buffers: made anew

    def _forms(self):
        """Type and shape of every buffer as the plan lays them out (the workspace's size is the plan's own)."""
        import torch
        s = self.shp
        i32, bf = torch.int32, torch.bfloat16
        per_token, per_request = (s.B, s.N), (s.B,)
        lat_e, rows_q, rows = (s.B, s.ne_cap, s.C), (s.B, s.q_cap, s.H, s.D), (s.B, s.n_full, s.H, s.D)
        return dict(mask=(torch.uint8, per_token), edit_idx=(i32, per_token), keep_idx=(i32, per_token),
                    slot=(i32, per_token), n_edit=(i32, per_request), n_q=(i32, per_request), n_cache=(i32, per_request),
                    n_rows=(i32, per_request), query_rows=(i32, (s.B, s.q_cap)), cache_rows=(i32, (s.B, s.n_full)),
                    x_e=(bf, lat_e), v_e=(bf, lat_e), v_avd=(bf, lat_e), x_out=(bf, (s.B, s.N, s.C)), q_e=(bf, rows_q),
                    k_fresh=(bf, rows_q), v_fresh=(bf, rows_q), k_cache=(bf, rows), v_cache=(bf, rows), o_full=(bf, rows))

    def _new_plan(self):
        s = self.shp
        return binding.StepPlan(s.B, s.N, s.n_text, s.n_ref, s.C, s.H, s.D, s.ne_cap, int(s.metric), int(s.membership),
                                float(s.threshold))

    def _step_plan(self):
        """The plan of the one-call step, or None where a buffer is not of the form it stands for.  It holds addresses,
        so it is compared with the buffers and the sizes as they are now, and made anew when one of them has changed."""
        s, d = self.shp, self.__dict__
        of = ([None if d[n] is None else d[n].data_ptr() for n in self._BUFFERS],
              (s.B, s.N, s.n_text, s.n_ref, s.C, s.H, s.D, s.ne_cap, s.membership))
        if self._plan_of != of:
            plan = None
            if all(d[n] is not None and d[n].is_cuda and d[n].dtype == dtype and tuple(d[n].shape) == shape and
                   d[n].is_contiguous() for n, (dtype, shape) in self._forms().items()) and \
               all(d[n] is None or d[n].is_cuda and d[n].is_contiguous() for n in ("workspace", "dev_status")):
                plan = self._new_plan()
                for name, at in zip(self._BUFFERS, of[0]):
                    setattr(plan, name, at)
                ws = self.workspace
                plan.workspace_bytes = 0 if ws is None else ws.numel() * ws.element_size()
            object.__setattr__(self, "_plan", plan)
            object.__setattr__(self, "_plan_of", of)
        if self._plan is not None:
            self._plan.metric, self._plan.threshold = int(s.metric), s.threshold
        return self._plan

    def run(self, x_t, v, ref, q_full, k_full, v_full, t, scale, dt, dt_unedited, stream=None,
            store_cache=True):
        """One region-aware step.  ``store_cache=False`` leaves the cache as the last storing call wrote
        it (Algorithm 1 refreshes it at full steps only; valid while the partition is unchanged)."""
        args = (x_t, v, ref, q_full, k_full, v_full, t, scale, dt, dt_unedited, store_cache)
        plan, B, events, before = self._step_plan(), binding, self.attention_events, binding.kernel_launches()
        if plan is None:
            return self._run_calls(*args, stream)
        try:
            B.region_step(plan, *args, parts=B.STEP_MOVES | (0 if events else B.STEP_ATTENTION), stream=stream)
        except B.ShapeError:                             # (nothing has been launched)
            s, rows = self.shp, lambda t: len(t.shape) > 2 and t.shape[0] == s.B and t.shape[2:].numel() == s.H * s.D
            if x_t.shape != (s.B, s.N, s.C) or v.shape != x_t.shape or ref.numel() != x_t.numel() or \
                    not (rows(q_full) and rows(k_full) and rows(v_full)):
                raise
            return self._run_calls(*args, stream)
        if events:
            events[0].record(stream)
            B.region_step(plan, *args, parts=B.STEP_ATTENTION, stream=stream)
            events[1].record(stream)
        self.launches += 8 if store_cache else 7
        self.kernel_launches += B.kernel_launches() - before
        return self.x_out

    # buffers that may hold another number of rows per request than planned, those that share it together
    _ROWS = (("x_e", "v_e", "v_avd"), ("q_e", "k_fresh", "v_fresh", "query_rows"), ("k_cache", "v_cache", "cache_rows"),
             ("o_full",))

    def _check_shapes(self):
        free = {n: group[0] for group in self._ROWS for n in group}
        for n, (_, shape) in self._forms().items():
            got = tuple(getattr(self, n).shape)
            if n in free and len(got) == len(shape) and (n != "cache_rows" or self.shp.B > 1):
                shape = (shape[0], getattr(self, free[n]).shape[1], *shape[2:])
            if got != shape and (n != "cache_rows" or len(got) != 2 or got[0] != shape[0] or self.shp.B > 1):
                raise binding.RegionEError(f"{n} must have shape {shape}, got {got}")

    def _run_calls(self, x_t, v, ref, q_full, k_full, v_full, t, scale, dt, dt_unedited, store_cache, stream):
        """The step as separate library calls, which take their sizes from the tensors: for inputs and buffers of other
        shapes than the plan's (rows as one dimension, a larger output, a cache that holds fewer rows)."""
        s, st, b, before = self.shp, self.dev_status, binding, binding.kernel_launches()
        self._check_shapes()
        b.partition_rows(x_t, v, ref, t, s.metric, s.threshold, self.mask, self.edit_idx, self.keep_idx, self.slot,
                         self.n_edit, s.n_text, s.n_ref, s.membership, self.query_rows, self.n_q, self.cache_rows,
                         self.n_cache, dev_status=st, stream=stream)
        b.gather_multi([x_t, v], self.edit_idx, self.n_edit, [self.x_e, self.v_e], dev_status=st, stream=stream)
        b.velocity_decay(self.v_e, scale, dt, self.x_e, self.n_edit, v_cache_out=self.v_avd, dev_status=st, stream=stream)
        b.merge(x_t, v, self.x_e, self.slot, dt_unedited, self.x_out, dev_status=st, stream=stream)
        if store_cache:
            b.rikv_store(k_full, v_full, self.cache_rows, self.n_cache, self.k_cache, self.v_cache, dev_status=st,
                         stream=stream)
        b.gather_multi([q_full, k_full, v_full], self.query_rows, self.n_q, [self.q_e, self.k_fresh, self.v_fresh],
                       dev_status=st, stream=stream)
        if self.attention_events is not None:
            self.attention_events[0].record(stream)
        b.region_attention_scatter(self.q_e, self.k_fresh, self.v_fresh, self.k_cache, self.v_cache, self.n_q, self.n_q,
                                   self.n_cache, self.o_full, self.query_rows, workspace=self.workspace, dev_status=st,
                                   stream=stream)
        if self.attention_events is not None:
            self.attention_events[1].record(stream)
        self.launches += 8 if store_cache else 7
        self.kernel_launches += b.kernel_launches() - before
        return self.x_out
