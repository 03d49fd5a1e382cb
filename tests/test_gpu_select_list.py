"""GPU: the list selection at the edges of its rounds, slices and clusters, on scores with ties, plateaus, zeros and hostile
orderings, against an exact sort of the scores it reports."""
import numpy as np
import pytest
import torch

from oracle import slkv_oracle as O
from paper_2508_15806_b200 import binding as B

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


def run(lens, hkv, w, budgets, pool, mode, k_scale=1.0, k_fn=None):
    d, T = 64, sum(lens)
    g = torch.Generator(device=DEV).manual_seed(sum(lens) + pool)
    q = torch.randn(len(lens), w, hkv, d, generator=g, device=DEV).bfloat16()
    k = (torch.randn(T, hkv, d, generator=g, device=DEV) * k_scale)
    k = (k if k_fn is None else k_fn(k)).bfloat16()
    cu = np.concatenate([[0], np.cumsum(lens)]).tolist()
    p = B.make_params(q, k, k, w, pool, mode)
    bud = torch.tensor(budgets, dtype=torch.int32, device=DEV)
    cap = sum(min(n, max(b, w)) for n in lens for b in budgets)
    out = torch.zeros(cap, d, dtype=torch.bfloat16, device=DEV)
    off = torch.zeros(len(lens) * hkv + 1, dtype=torch.int32, device=DEV)
    kept = torch.full((cap,), -1, dtype=torch.int32, device=DEV)
    pooled = torch.zeros(max(B.slkv_pooled_elems(p, cu), 1), device=DEV)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    ws = torch.empty(B.slkv_workspace_bytes(p, cu), dtype=torch.uint8, device=DEV)
    for want in (pooled, None):                         # the same with and without the scores written out
        kept.fill_(-1)
        B.slkv_compress(p, q, k, k, torch.tensor(cu, dtype=torch.int32, device=DEV), cu, bud, out, torch.zeros_like(out), off,
                        kept, ws, want, status)
        torch.cuda.synchronize()
        assert int(status) == 0
        sc, idx, o, at = pooled.cpu().numpy(), kept.cpu().numpy(), off.cpu().tolist(), 0
        for s, n in enumerate(lens):
            nh = max(n - w, 0)
            for h in range(hkv):
                seg = s * hkv + h
                kh, nw = O.kept_counts(n, budgets[h], w)
                ref = O.select_topk(sc[at:at + nh].astype(np.float64), kh) if kh else np.zeros(0, np.int64)
                got = idx[o[seg]:o[seg + 1]]
                assert got[:kh].tolist() == ref.tolist(), (s, h)
                assert got[kh:].tolist() == list(range(n - nw, n))
                at += nh


@pytest.mark.parametrize("n", [1, 3, 5, 127, 128, 4095, 4096, 4097, 8190, 32764, 32765, 32768, 40001, 131071])
@pytest.mark.parametrize("pool,mode", [(1, B.SLKV_POOL_MAX), (7, B.SLKV_POOL_MAX), (9, B.SLKV_POOL_AVG)])
def test_lengths(n, pool, mode):
    run([n + 8], 3, 8, [8 + max(1, n // 50), 8 + n // 2, 8 + n - 1], pool, mode)


def test_ragged_segments_start_anywhere():
    run([4100, 9, 8, 0, 700, 33001, 2], 3, 8, [40, 500, 9], 5, B.SLKV_POOL_MAX)


@pytest.mark.parametrize("n", [6000, 70000])
def test_ties_zeros_and_orderings(n):
    same = lambda k: k[:1].expand_as(k).contiguous()                                             # noqa: E731
    far = lambda k: torch.where(torch.arange(len(k), device=DEV).view(-1, 1, 1) % 97 == 0, k * 0.0 + 30.0, k * 0.0 - 30.0)   # noqa: E731
    sort = lambda k: torch.sort(k, dim=0).values                                                 # noqa: E731
    period = lambda k: k[torch.arange(len(k), device=DEV) % 128]                                 # noqa: E731
    for fn in (same, far, sort, period):
        run([n], 3, 4, [300, n // 3, n - 7], 3, B.SLKV_POOL_MAX, k_fn=fn)


@pytest.mark.parametrize("n", [2045, 2048, 2049, 4093, 4097, 8189, 8193, 16381, 16385])
@pytest.mark.parametrize("many", [False, True])
def test_edges_of_the_variants(n, many):
    # few CTAs (an SM each), and more of them than SMs; a short sequence in between moves the segments off 16-byte boundaries
    run(([n + 8] + [8 + 9] * 60 + [n + 8]) if many else [n + 8], 3, 8, [8 + max(1, n // 50), 8 + n // 2, 8 + n - 1], 7, B.SLKV_POOL_MAX)


@pytest.mark.parametrize("n", [8192, 16000, 32768, 70000])
@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_a_sample_that_misleads(n, sign):
    # every 16th (32nd) position is the one that is sampled: those positions high, or low, and the rest the other way
    for step in (16, 32):
        odd = lambda k: torch.where(torch.arange(len(k), device=DEV).view(-1, 1, 1) % step == step // 2, k * 0.05 + sign, k * 0.05 - sign)   # noqa: E731,B023
        run([n + 4], 3, 4, [300, n // 4, n - n // 10], 1, B.SLKV_POOL_MAX, k_fn=odd)


def short_keys(kind):
    """Keys of a segment whose scores share first-level bins: all equal, nearly uniform, in runs, in a trend, or all but a few so
    small (below 2^-24) that the lowest bin holds them."""
    at = lambda k: torch.arange(len(k), device=DEV)                                              # noqa: E731
    return {"equal": lambda k: k[:1].expand_as(k).contiguous(), "flat": lambda k: k * 0.1, "flatter": lambda k: k * 0.01,
            "periodic": lambda k: k[at(k) % 7], "pairs": lambda k: k[at(k) // 2] * 0.1,
            "ordered": lambda k: torch.sort(k, dim=0).values * 0.2,
            "tiny": lambda k: torch.where(at(k).view(-1, 1, 1) < 32, k * 40.0, k)}[kind]


@pytest.mark.parametrize("n", [200, 255, 256, 257, 258, 300, 400, 511, 512, 513, 600, 768, 1000, 1020, 1021, 1022])
@pytest.mark.parametrize("kind", ["equal", "flat", "flatter", "periodic", "pairs", "ordered", "tiny"])
def test_short_segments_in_one_bin(n, kind):
    for pool in (1, 7):
        run([n + 4], 3, 4, [4 + n // 10, 4 + n // 2, n + 1], pool, B.SLKV_POOL_MAX, k_fn=short_keys(kind))
    run([n + 4], 3, 4, [4 + n // 10, 4 + n // 2, n + 1], 5, B.SLKV_POOL_AVG, k_fn=short_keys(kind))


@pytest.mark.parametrize("n", [256, 257, 400, 512, 513, 1000])
@pytest.mark.parametrize("kind", ["equal", "flat", "tiny"])
def test_short_segments_of_many_rows_and_in_lists(n, kind):
    # 160 query rows per KV head, which only the list kernels take; one call, and a list of three layers
    w, hq, hkv, d, pool = 40, 8, 2, 64, 5
    g = torch.Generator(device=DEV).manual_seed(n)
    q = torch.randn(1, w, hq, d, generator=g, device=DEV).bfloat16()
    ks = [short_keys(kind)(torch.randn(n + w, hkv, d, generator=g, device=DEV)).bfloat16() for _ in range(3)]
    p, cu, budgets = B.make_params(q, ks[0], ks[0], w, pool), [0, n + w], [w + n // 8, w + n - 3]
    cap = sum(budgets)
    cu_dev, bud = torch.tensor(cu, dtype=torch.int32, device=DEV), torch.tensor(budgets, dtype=torch.int32, device=DEV)
    ws = torch.empty(B.slkv_workspace_bytes_overlapped(p, cu), dtype=torch.uint8, device=DEV)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    for call, layers in ((B.slkv_compress, ks[:1]), (B.slkv_compress_overlapped, ks)):
        res = []
        for k in layers:
            out = torch.zeros(2, cap, d, dtype=torch.bfloat16, device=DEV)
            off, kept = torch.zeros(hkv + 1, dtype=torch.int32, device=DEV), torch.full((cap,), -1, dtype=torch.int32, device=DEV)
            pooled = torch.zeros(B.slkv_pooled_elems(p, cu), device=DEV)
            call(p, q, k, k, cu_dev, cu, bud, out[0], out[1], off, kept, ws, pooled, status)
            res.append((pooled, kept, off, out))                   # a list writes them when it goes out
        B.slkv_join()
        torch.cuda.synchronize()
        assert int(status) == 0
        for pooled, kept, off, _ in res:
            sc, o = pooled.cpu().numpy().astype(np.float64), off.tolist()
            for h in range(hkv):
                ref = O.select_topk(sc[h * n:(h + 1) * n], budgets[h] - w)
                assert kept[o[h]:o[h + 1]].tolist() == ref.tolist() + list(range(n, n + w)), h
