"""Context-parallel compression of ONE long sequence (Sec. 3.4, Eq. 7-8; Algorithm 3): the per-rank call sequence of
the slkv_cp_* entry points with the collectives between them.

The history keys are split over the ranks by contiguous ranges; the last rank also holds the window rows.  Every step
of the arithmetic runs in the library's kernels; this module slices the rank's views, allocates its buffers and calls
the three kinds of collective the method needs per layer:
    all-gather of the rows' local log-sum-exps   [n_q_heads, window] float32
    3 x all-reduce (sum) of a radix histogram    [n_kv_heads, 2048] int32
    all-gather of the tie counts                 [n_kv_heads] int32
`comm` is anything with rank, world, all_gather(tensor) -> [world, ...] and all_reduce_sum(tensor) (in place):
DistComm wraps torch.distributed (NCCL for CUDA tensors, gloo for CPU tensors); tests emulate several ranks on one GPU
with a thread-and-barrier comm of their own.
"""
from __future__ import annotations

from dataclasses import dataclass
from typing import List, Optional, Sequence, Tuple

import torch

from . import binding as B


def key_ranges(seq_len: int, window: int, world: int) -> List[Tuple[int, int]]:
    """History positions [b, e) of every rank: the n_hist = seq_len - window history keys in `world` near-equal
    contiguous shares (the first n_hist % world ranks hold one more); the last rank also holds the window rows."""
    n_hist = max(seq_len - window, 0)
    base, extra = divmod(n_hist, world)
    out, b = [], 0
    for r in range(world):
        e = b + base + (1 if r < extra else 0)
        out.append((b, e))
        b = e
    return out


class DistComm:
    """torch.distributed as the communicator (one process per GPU; NCCL moves CUDA tensors, gloo CPU tensors)."""

    def __init__(self, group=None):
        import torch.distributed as dist
        self._dist, self._group = dist, group
        self.rank, self.world = dist.get_rank(group), dist.get_world_size(group)

    def all_gather(self, t: torch.Tensor) -> torch.Tensor:
        out = torch.empty(self.world * t.numel(), dtype=t.dtype, device=t.device)
        self._dist.all_gather_into_tensor(out, t.contiguous().reshape(-1), group=self._group)
        return out.reshape((self.world,) + tuple(t.shape))

    def all_reduce_sum(self, t: torch.Tensor) -> torch.Tensor:
        self._dist.all_reduce(t, op=self._dist.ReduceOp.SUM, group=self._group)
        return t


@dataclass
class RankShard:
    """What one rank holds of a layer: q_win [1, window, n_q_heads, d]; k, v [rows, n_kv_heads, d] = the history
    positions [begin - margin_left, end + margin_right) and, on the last rank, the window rows behind them."""
    rank: int
    world: int
    seq_len: int
    window: int
    begin: int
    end: int
    margin_left: int
    margin_right: int
    q_win: torch.Tensor
    k: torch.Tensor
    v: torch.Tensor

    @property
    def last(self) -> bool:
        return self.rank == self.world - 1

    @property
    def own(self) -> int:
        return self.end - self.begin


def shard_of(q_win: torch.Tensor, k: torch.Tensor, v: torch.Tensor, window: int, pool_kernel: int, rank: int,
             world: int) -> RankShard:
    """The rank's views of a whole sequence's q_win [1, w, Hq, d], k, v [seq_len, Hkv, d] (for callers and tests that
    hold the whole sequence; a context-parallel prefill already holds each rank's rows and fills RankShard itself)."""
    seq_len = k.shape[0]
    n_hist = max(seq_len - window, 0)
    b, e = key_ranges(seq_len, window, world)[rank]
    ml = min(pool_kernel // 2, b)
    mr = 0 if rank == world - 1 else min(pool_kernel // 2, n_hist - e)
    hi = seq_len if rank == world - 1 else e + mr
    return RankShard(rank, world, seq_len, window, b, e, ml, mr, q_win, k[b - ml:hi], v[b - ml:hi])


def compress_rank(shard: RankShard, budgets_row: torch.Tensor, pool_kernel: int, comm, pool_mode: int = B.SLKV_POOL_MAX,
                  softmax_domain: int = B.SLKV_HISTORY, score_path: int = B.SLKV_PATH_AUTO, stream=None) -> dict:
    """One layer on one rank.  budgets_row: CUDA int32 [n_kv_heads], the layer's budgets (the same on every rank).
    Returns this rank's packed rows: k_out, v_out [capacity, d], offsets [n_kv_heads + 1] (local), kept_idx (positions
    in the whole sequence), status, pooled (the rank's scores, margins included) and lse (the merged row statistics)."""
    sh = shard
    assert sh.seq_len >= sh.window and comm.world == sh.world and comm.rank == sh.rank
    dev, dt = sh.k.device, sh.k.dtype
    w, own, (rows, hkv, d), hq = sh.window, sh.own, sh.k.shape, sh.q_win.shape[2]
    n_win = w if sh.last else 0
    n_ext = sh.margin_left + own + sh.margin_right
    row_stride, cap = max(n_ext, 1), hkv * (own + n_win)
    p = B.make_params(sh.q_win, sh.k, sh.v, w, pool_kernel, pool_mode, score_path, softmax_domain, B.SLKV_LSE_LOG2)
    p.history_only = 0 if sh.last else 1

    # One buffer for all scratch, zero at the start: what the steps add to (row sums, histograms, totals).  Another for the small
    # outputs, which a caller keeps without any scratch, and without the scores.  One call clears both, in front of all steps.
    n_own = own + n_win
    has_keys = own > 0 or (sh.last and softmax_domain == B.SLKV_ALL_CAUSAL)
    ws_score = B.slkv_workspace_bytes(p, (0, rows)) if n_ext > 0 else 0
    ws_lse = 0 if not has_keys else (ws_score if n_own == rows and n_ext > 0 else B.slkv_workspace_bytes(p, (0, n_own)))
    ws_emit = B.slkv_cp_workspace_bytes(hkv, own, max(cap, 1))
    state_bytes = -(-32 * hkv // 256) * 256                    # [4][2][hkv]: every head's prefix and need after each level
    sizes = ((state_bytes + max(ws_score, ws_lse, ws_emit)) // 4, 3 * 2048 * hkv, hkv, hkv, hq * w)
    out_sizes = (max(cap, 1), hq * w, hkv + 1, 1)
    buf, out = torch.empty(sum(sizes), dtype=torch.int32, device=dev), torch.empty(sum(out_sizes), dtype=torch.int32, device=dev)
    torch._foreach_zero_((buf, out))
    ws, hists, totals, ties, lse_local = buf.split(sizes)
    kept_idx, lse, offsets, status = out.split(out_sizes)
    pooled = (torch.empty if n_ext > 0 else torch.zeros)(hkv * row_stride, dtype=torch.float32, device=dev)
    state = ws.data_ptr()
    scratch = state + state_bytes
    lse_local, lse = lse_local.view(torch.float32).view(hq, w), lse.view(torch.float32).view(1, hq, w)

    # 1. the rows' log-sum-exp over the keys this rank owns (the last rank's range is an ordinary sequence tail)
    if has_keys:
        k_own = sh.k if n_own == rows else sh.k[sh.margin_left:sh.margin_left + n_own]
        B.slkv_cp_row_lse(p, sh.q_win, k_own, status, (0, n_own), lse_local, scratch, ws_lse, status, stream)
    else:
        lse_local.fill_(float("-inf"))
    # 2. merged over the ranks
    B.slkv_cp_merge_lse(p, comm.all_gather(lse_local), lse, stream)
    # 3. pooled scores of the owned rows and the neighbours' margins
    if n_ext > 0:
        B.slkv_score_at(p, sh.q_win, sh.k, status, (0, rows), pooled, scratch, ws_score, status, stream, lse)
    # 4. every head's threshold: radix descent on histograms summed over the ranks; the output rows are cleared meanwhile,
    #    a quarter beside each level (every row is whole 16-byte units)
    out_k, out_v = torch.empty(2, max(cap, 1), d, dtype=dt, device=dev).unbind(0)
    clear, all16 = out_k.data_ptr(), 2 * out_k.numel() * out_k.element_size() // 16
    hist_sum = None
    for level, hist in enumerate((*hists.view(3, hkv, 2048).unbind(0), None)):
        b, e = all16 * level // 4, all16 * (level + 1) // 4
        B.slkv_cp_step(budgets_row, hkv, w, sh.seq_len, level, state, hist_sum, pooled, row_stride, sh.margin_left, own,
                       hist, totals, clear + 16 * b, 16 * (e - b), scratch, ws_emit, stream)
        if hist is not None:
            comm.all_reduce_sum(hist)
        hist_sum = hist
    # 5. ties in rank order, then this rank's packed rows
    ties_all = comm.all_gather(ties)
    threshold = state + 24 * hkv
    B.slkv_cp_emit_counted(p, sh.k, sh.v, rows, pooled, row_stride, sh.margin_left, own, sh.begin, threshold,
                           threshold + 4 * hkv, ties_all, sh.rank, n_win, sh.seq_len - n_win, totals, out_k, out_v,
                           offsets, kept_idx, scratch, ws_emit, status, stream)
    return dict(k_out=out_k, v_out=out_v, offsets=offsets, kept_idx=kept_idx, status=status, pooled=pooled, lse=lse,
                capacity=cap, keep_alive=(buf, ties_all))


def stitch_heads(per_rank: Sequence[dict], n_kv_heads: int) -> List[dict]:
    """Per KV head, the whole sequence's packed cache from the ranks' outputs (rank order = position order): for
    callers that bring the ranks' rows together, and for tests.  Returns [{"kept_idx", "k", "v"}] per head."""
    heads = []
    for h in range(n_kv_heads):
        idx, ks, vs = [], [], []
        for o in per_rank:
            a, b = int(o["offsets"][h]), int(o["offsets"][h + 1])
            idx.append(o["kept_idx"][a:b])
            ks.append(o["k_out"][a:b])
            vs.append(o["v_out"][a:b])
        heads.append(dict(kept_idx=torch.cat(idx), k=torch.cat(ks), v=torch.cat(vs)))
    return heads
