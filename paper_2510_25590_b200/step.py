"""One region-aware denoising step for one attention layer, as one C-ABI call.

This is buffer ownership only (torch tensors are device buffers): every operation runs in the
library's kernels.  The sequence follows Algorithm 1 of the paper for one layer:

  partition with the joint-sequence row lists -> gather X^E, v^E; velocity decay + Euler update; merge with
  the one-step-predicted unedited tokens; gather of the recomputed rows of Q (K, V) -> region attention
  writing its rows back at their joint-sequence positions, the RIKV store in the same launch

(four kernel launches: partition, moves, attention, merge of the attention's shared items).

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
        self.workspace = None
        self.workspace = torch.empty(max(binding.region_step_workspace(self._step_plan()), 256), dtype=torch.uint8,
                                     device=device)
        self.launches = 0                 # operations of the sequence run so far (8 per step, 7 without the store)
        self.kernel_launches = 0          # kernels launched so far, at least (a fourth merges cut items in some shapes)
        self.attention_events = None      # optional (start, stop) pair recorded around the attention

    _BUFFERS = ("mask", "edit_idx", "keep_idx", "slot", "n_edit", "query_rows", "n_q", "cache_rows", "n_cache", "n_rows",
                "x_e", "v_e", "v_avd", "x_out", "q_e", "k_fresh", "v_fresh", "k_cache", "v_cache", "o_full", "workspace",
                "dev_status")

    def __setattr__(self, name, value):
        object.__setattr__(self, name, value)
        if name in self._BUFFERS or name == "shp":
            object.__setattr__(self, "_plan", None)      # the plan names this object's buffers: made anew

    def _step_plan(self):
        if self._plan is None:
            s = self.shp
            p = binding.StepPlan(s.B, s.N, s.n_text, s.n_ref, s.C, s.H, s.D, s.ne_cap, int(s.metric), int(s.membership),
                                 float(s.threshold))
            for name in self._BUFFERS:
                t = getattr(self, name)
                setattr(p, name, None if t is None else t.data_ptr())
            p.workspace_bytes = 0 if self.workspace is None else self.workspace.numel()
            object.__setattr__(self, "_plan", p)
        self._plan.metric, self._plan.threshold = int(self.shp.metric), self.shp.threshold
        return self._plan

    def run(self, x_t, v, ref, q_full, k_full, v_full, t, scale, dt, dt_unedited, stream=None,
            store_cache=True):
        """One region-aware step.  ``store_cache=False`` leaves the cache as the last storing call wrote
        it (Algorithm 1 refreshes it at full steps only; valid while the partition is unchanged)."""
        args = (self._step_plan(), x_t, v, ref, q_full, k_full, v_full, t, scale, dt, dt_unedited, store_cache)
        if self.attention_events is None:
            binding.region_step(*args, stream=stream)
        else:
            binding.region_step(*args, parts=binding.STEP_MOVES, stream=stream)
            self.attention_events[0].record(stream)
            binding.region_step(*args, parts=binding.STEP_ATTENTION, stream=stream)
            self.attention_events[1].record(stream)
        self.launches += 8 if store_cache else 7
        self.kernel_launches += 3
        return self.x_out
