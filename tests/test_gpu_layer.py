"""GPU: single calls that do the whole layer in one launch (a cluster of CTAs per segment), against the general path launch by
launch -- which a call that asks for the pooled scores takes -- and the scores alone against the oracle."""
import numpy as np
import pytest
import torch

import parity as P
from oracle import slkv_oracle as O
from paper_2508_15806_b200 import binding as B

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


def inputs(seed, lens, hq, hkv, d, w, dt=torch.bfloat16, scale=1.0):
    g = torch.Generator(device=DEV).manual_seed(seed)
    T = sum(lens)
    q, k, v = (torch.randn(*s, generator=g, device=DEV) for s in ((len(lens), w, hq, d), (T, hkv, d), (T, hkv, d)))
    return (q * scale).to(dt), (k * scale).to(dt), v.to(dt), np.concatenate([[0], np.cumsum(lens)]).tolist()


def both(q, k, v, cu, w, pool, budgets, mode=B.SLKV_POOL_MAX, domain=B.SLKV_HISTORY, lse=None, cap=None, one_launch=True, calls=1):
    """(one launch, general path): offsets, kept positions, rows."""
    p = B.make_params(q, k, v, w, pool, mode, softmax_domain=domain, lse_units=B.SLKV_LSE_LOG2)
    hkv, d, n = k.shape[1], k.shape[2], len(cu) - 1
    bud = torch.tensor(budgets, dtype=torch.int32, device=DEV)
    cap = cap if cap is not None else max(sum(min(b - a, max(c, w)) for a, b in zip(cu, cu[1:]) for c in budgets), 1)
    cu_dev = torch.tensor(cu, dtype=torch.int32, device=DEV)
    ws = torch.empty(B.slkv_workspace_bytes(p, cu), dtype=torch.uint8, device=DEV)
    res = []
    for pooled in (None, torch.zeros(max(B.slkv_pooled_elems(p, cu), 1), device=DEV)):
        ko, vo = (torch.zeros(max(cap, 1), d, dtype=k.dtype, device=DEV) for _ in range(2))
        off, kept = torch.full((n * hkv + 1,), -1, dtype=torch.int32, device=DEV), torch.full((max(cap, 1),), -1, dtype=torch.int32, device=DEV)
        status = torch.zeros(1, dtype=torch.int32, device=DEV)
        for _ in range(calls):
            B.slkv_compress(p, q, k, v, cu_dev, cu, bud, ko[:cap], vo[:cap], off, kept, ws, pooled, status, lse=lse)
        if pooled is None:
            assert not one_launch or B.slkv_last_launch_count() == 1
        torch.cuda.synchronize()
        res.append((off, kept, ko, vo, status))
    return res


def same(res, status=0):
    a, b = res
    assert int(a[4]) == status and int(b[4]) == status
    for x, y in zip(a[:4], b[:4]):
        assert torch.equal(x, y)


@pytest.mark.parametrize("hq,hkv,d,w", [(8, 8, 128, 1), (8, 4, 64, 16), (32, 8, 128, 32), (5, 1, 64, 25), (24, 8, 128, 32)])
@pytest.mark.parametrize("n", [1, 127, 128, 129, 1023, 1025, 2000, 4096, 4097, 8191, 8192])
def test_lengths(hq, hkv, d, w, n):
    q, k, v, cu = inputs(n + hq, [n + w], hq, hkv, d, w)
    same(both(q, k, v, cu, w, 7, [(0, w, w + 1, w + n // 3, w + n - 1, w + n, w + n + 9, w + 64)[h] for h in range(hkv)]))


@pytest.mark.parametrize("lens", [[3000, 0, 31, 32, 33, 700], [160, 1100] * 4, [300] * 8])
@pytest.mark.parametrize("mode,pool", [(B.SLKV_POOL_MAX, 1), (B.SLKV_POOL_AVG, 5), (B.SLKV_POOL_AVG, 9), (B.SLKV_POOL_MAX, 3)])
def test_ragged_batches(lens, mode, pool):
    q, k, v, cu = inputs(len(lens) + pool, lens, 16, 4 if len(lens) == 6 else 8, 64, 32)
    same(both(q, k, v, cu, 32, pool, [40, 300, 33, 5000][:k.shape[1]] * (k.shape[1] // 4), mode))


@pytest.mark.parametrize("d,w,hq,hkv,n", [(64, 32, 32, 8, 4061), (128, 17, 4, 4, 900), (128, 64, 2, 1, 2500), (64, 100, 2, 2, 4000)])
def test_domains_and_supplied_statistics(d, w, hq, hkv, n):
    q, k, v, cu = inputs(d + w, [n + w], hq, hkv, d, w)
    bud = [w + 10 + 50 * h for h in range(hkv)]
    same(both(q, k, v, cu, w, 5, bud, domain=B.SLKV_ALL_CAUSAL))
    p = B.make_params(q, k, v, w, 5, softmax_domain=B.SLKV_ALL_CAUSAL, lse_units=B.SLKV_LSE_LOG2)
    lse = torch.zeros(1, hq, w, device=DEV)
    ws = torch.empty(B.slkv_workspace_bytes(p, cu), dtype=torch.uint8, device=DEV)
    cu_dev = torch.tensor(cu, dtype=torch.int32, device=DEV)
    B.slkv_row_lse(p, q, k, cu_dev, cu, lse, ws)
    same(both(q, k, v, cu, w, 5, bud, lse=lse))
    # the scores alone, with the library's statistics and with the same handed in
    own, fed = (torch.zeros(B.slkv_pooled_elems(p, cu), device=DEV) for _ in range(2))
    B.slkv_score(p, q, k, cu_dev, cu, own, ws)
    assert B.slkv_last_launch_count() == 1
    B.slkv_score(p, q, k, cu_dev, cu, fed, ws, lse=lse)
    assert torch.equal(own, fed)
    ref = P.oracle_pooled(q.cpu(), k.cpu(), cu, w, 5, domain=B.SLKV_ALL_CAUSAL)
    P.assert_pooled_close(own.cpu().numpy(), ref, cu, hkv, w)


def test_scores_beyond_fp32_and_fp64():
    # log-sum-exps of up to some 6000 in log2 units are rounded to 2^-11, which a vote shows as 2^-11 ln 2 of its value, twice
    for scale, shift in ((6.0, 40.0), (40.0, 300.0)):
        q, k, v, cu = inputs(3, [1500], 8, 2, 128, 32, scale=scale)
        k[:, :, 0] += shift
        q[:, :16, :, 0], q[:, 16:, :, 0] = 80.0, -80.0
        p = B.make_params(q, k, v, 32, 7)
        one, general = (torch.zeros(B.slkv_pooled_elems(p, cu), device=DEV) for _ in range(2))
        status = torch.zeros(1, dtype=torch.int32, device=DEV)
        cu_dev, bud = torch.tensor(cu, dtype=torch.int32, device=DEV), torch.tensor([100, 200], dtype=torch.int32, device=DEV)
        ws = torch.empty(B.slkv_workspace_bytes(p, cu), dtype=torch.uint8, device=DEV)
        B.slkv_score(p, q, k, cu_dev, cu, one, ws, status)
        assert int(status) == 0 and B.slkv_last_launch_count() == 1
        out = torch.zeros(300, 128, dtype=torch.bfloat16, device=DEV)
        B.slkv_compress(p, q, k, v, cu_dev, cu, bud, out, torch.zeros_like(out), torch.zeros(3, dtype=torch.int32, device=DEV),
                        torch.zeros(300, dtype=torch.int32, device=DEV), ws, general, status)
        assert int(status) == 0 and torch.isfinite(one).all() and (one > 0).any()
        assert torch.allclose(one, general, rtol=7e-4, atol=1e-30)


def test_views_and_capacity():
    # K and V slices of one fused buffer, heads outermost; then too little room
    w, n, hkv, d = 32, 1900, 4, 128
    q, _, _, cu = inputs(5, [n], 16, hkv, d, w)
    kv = torch.randn(2 * hkv, n + 5, d, device=DEV).bfloat16()
    k, v = kv[:hkv, 5:].transpose(0, 1), kv[hkv:, 5:].transpose(0, 1)
    qt = q.permute(0, 2, 1, 3).contiguous().permute(0, 2, 1, 3)
    for qq in (q, qt):
        same(both(qq, k, v, cu, w, 7, [100, 1500, 33, 64]))
    same(both(q, k, v, cu, w, 7, [100, 1500, 33, 64], cap=777), status=B.ERR["CAPACITY"])
    same(both(q, k, v, cu, w, 7, [100, 1500, 33, 64], cap=1), status=B.ERR["CAPACITY"])


@pytest.mark.parametrize("n", [1500, 8192])
def test_many_calls_in_a_row(n):
    # 8192 positions: a CTA's tiles go round the ring of K tiles, and come back for the votes
    q, k, v, cu = inputs(n, [n + 32], 32, 8, 128, 32)
    same(both(q, k, v, cu, 32, 7, [64 + 100 * h for h in range(8)], calls=1000))


@pytest.mark.parametrize("lens", [[100], [300], [700], [1000], [1180], [40, 1100, 33, 200], [600, 34, 6000]])
def test_rows_of_ctas_without_tiles(lens):
    # Segments of fewer tiles than their cluster has CTAs, log-sum-exps handed in: a CTA without tiles gets to its rows with
    # nothing to wait for but the budgets, which another warp reads -- from HBM, while the log-sum-exps lie in L2.
    w, hq, hkv, d = 32, 8, 4, 64
    q, k, v, cu = inputs(sum(lens), lens, hq, hkv, d, w)
    p = B.make_params(q, k, v, w, 7, lse_units=B.SLKV_LSE_LOG2)
    cu_dev = torch.tensor(cu, dtype=torch.int32, device=DEV)
    ws = torch.empty(B.slkv_workspace_bytes(p, cu), dtype=torch.uint8, device=DEV)
    lse = torch.zeros(len(lens), hq, w, device=DEV)
    B.slkv_row_lse(p, q, k, cu_dev, cu, lse, ws)
    sweep = torch.empty(1 << 28, dtype=torch.uint8, device=DEV)
    rng = np.random.default_rng(sum(lens))
    for _ in range(40):
        budgets = rng.integers(1, max(lens) + 40, hkv).tolist()
        bud = torch.tensor(budgets, dtype=torch.int32, device=DEV)
        cap = sum(min(n, max(c, w)) for n in lens for c in budgets)
        res = []
        for pooled in (None, torch.zeros(B.slkv_pooled_elems(p, cu), device=DEV)):
            ko, vo = (torch.zeros(cap, d, dtype=k.dtype, device=DEV) for _ in range(2))
            off, kept = torch.full((len(lens) * hkv + 1,), -1, dtype=torch.int32, device=DEV), torch.full((cap,), -1, dtype=torch.int32, device=DEV)
            status = torch.zeros(1, dtype=torch.int32, device=DEV)
            sweep.zero_()
            lse.add_(0.0)
            B.slkv_compress(p, q, k, v, cu_dev, cu, bud, ko, vo, off, kept, ws, pooled, status, lse=lse)
            assert pooled is not None or B.slkv_last_launch_count() == 1
            res.append((off, kept, ko, vo, status))
        same(res)


# ---- fp32 -------------------------------------------------------------------------------------------------------------
def check_fp32(hq, hkv, d, w, lens, pool=5, mode=B.SLKV_POOL_MAX, domain=B.SLKV_HISTORY, q_fn=None, rtol=1e-5, one_launch=True):
    """Scores and row statistics of the one launch (without and with supplied statistics) against the general path's, the kept
    positions against an exact sort of the scores."""
    q, k, v, cu = inputs(hq + d + w + sum(lens), lens, hq, hkv, d, w, torch.float32)
    if q_fn:
        q_fn(q, k)
    p = B.make_params(q, k, v, w, pool, mode, softmax_domain=domain, lse_units=B.SLKV_LSE_LOG2)
    cu_dev = torch.tensor(cu, dtype=torch.int32, device=DEV)
    ws = torch.empty(B.slkv_workspace_bytes(p, cu), dtype=torch.uint8, device=DEV)
    lse = torch.zeros(len(lens), hq, w, device=DEV)
    own, fed, general = (torch.full((max(B.slkv_pooled_elems(p, cu), 1),), 7.0, device=DEV) for _ in range(3))
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    B.slkv_row_lse(p, q, k, cu_dev, cu, lse, ws, status)
    B.slkv_score(p, q, k, cu_dev, cu, own, ws, status)
    assert not one_launch or B.slkv_last_launch_count() == 1
    B.slkv_score(p, q, k, cu_dev, cu, fed, ws, status, lse=lse)
    assert torch.equal(own, fed)
    budgets = [w + 3 + 37 * h for h in range(hkv)]
    res = both(q, k, v, cu, w, pool, budgets, mode, domain, one_launch=one_launch)
    bud, cap = torch.tensor(budgets, dtype=torch.int32, device=DEV), res[0][2].shape[0]
    B.slkv_compress(p, q, k, v, cu_dev, cu, bud, torch.zeros(cap, d, device=DEV), torch.zeros(cap, d, device=DEV),
                    torch.zeros(len(lens) * hkv + 1, dtype=torch.int32, device=DEV), torch.zeros(cap, dtype=torch.int32, device=DEV), ws,
                    general, status)
    assert int(status) == 0 and torch.allclose(own, general, rtol=rtol, atol=1e-30)
    off, kept, ko, vo, st = res[0]
    assert int(st) == 0 and torch.equal(off, res[1][0])
    sc, at = own.cpu().numpy(), 0
    for s, n in enumerate(lens):
        nh = max(n - w, 0)
        for h in range(hkv):
            kh, nw = O.kept_counts(n, budgets[h], w)
            ref = O.select_topk(sc[at:at + nh].astype(np.float64), kh) if kh else np.zeros(0, np.int64)
            a, b = int(off[s * hkv + h]), int(off[s * hkv + h + 1])
            got = kept[a:b].cpu()
            assert got.tolist() == ref.tolist() + list(range(n - nw, n)), (s, h)
            assert torch.equal(ko[a:b], k[cu[s] + got.to(DEV).long(), h]) and torch.equal(vo[a:b], v[cu[s] + got.to(DEV).long(), h])
            at += nh


@pytest.mark.parametrize("hq,hkv,d,w", [(8, 8, 64, 16), (2, 2, 128, 1), (16, 8, 128, 16), (6, 2, 64, 21), (16, 4, 64, 32)])
@pytest.mark.parametrize("n", [1, 31, 32, 33, 319, 321, 400, 1008])
def test_fp32_lengths(hq, hkv, d, w, n):
    check_fp32(hq, hkv, d, w, [n + w])


@pytest.mark.parametrize("hq,hkv,d,w,n", [(8, 8, 64, 16, 5000), (8, 4, 128, 8, 8192), (4, 4, 128, 16, 4096), (4, 4, 64, 16, 4097), (32, 8, 128, 16, 2400)])
@pytest.mark.parametrize("domain", [B.SLKV_HISTORY, B.SLKV_ALL_CAUSAL])
def test_fp32_long(hq, hkv, d, w, n, domain):
    check_fp32(hq, hkv, d, w, [n + w], 7, domain=domain, one_launch=hkv == 8)


@pytest.mark.parametrize("mode,pool", [(B.SLKV_POOL_MAX, 1), (B.SLKV_POOL_AVG, 9)])
def test_fp32_ragged_batch(mode, pool):
    check_fp32(8, 4, 64, 32, [900, 0, 31, 32, 33, 1100], pool, mode, B.SLKV_ALL_CAUSAL)


def test_fp32_beyond_its_range():
    def far(q, k):
        k[:, :, 0] += 60.0
        q[:, :4, :, 0], q[:, 4:, :, 0] = 70.0, -70.0
    # log-sum-exps of some 750 in log2 units, rounded to 2^-14: a vote shows that twice
    for domain in (B.SLKV_HISTORY, B.SLKV_ALL_CAUSAL):
        check_fp32(4, 2, 64, 8, [900], domain=domain, q_fn=far, rtol=1e-4)


@pytest.mark.parametrize("hq,hkv,d,w", [(8, 8, 64, 16), (4, 2, 64, 5), (2, 1, 128, 17), (8, 4, 64, 33), (2, 1, 64, 64)])
@pytest.mark.parametrize("n", [300, 700, 735, 1400, 1450, 2600, 2740])
def test_fp32_equal_keys_have_equal_scores(hq, hkv, d, w, n):
    # The CTAs of a segment hold blocks of keys that differ by one in number, which the threads of a CTA share out differently:
    # a key's score is the same wherever it lies, bit for bit, and the same as the general path's.
    for domain, every in ((B.SLKV_HISTORY, 1), (B.SLKV_ALL_CAUSAL, 37)):
        q, k, v, cu = inputs(n + w, [n + w], hq, hkv, d, w, torch.float32)
        k[:n] = k[torch.arange(n, device=DEV) % every]
        p = B.make_params(q, k, v, w, 1, softmax_domain=domain)
        cu_dev, status = torch.tensor(cu, dtype=torch.int32, device=DEV), torch.zeros(1, dtype=torch.int32, device=DEV)
        ws = torch.empty(B.slkv_workspace_bytes(p, cu), dtype=torch.uint8, device=DEV)
        own, general = (torch.zeros(B.slkv_pooled_elems(p, cu), device=DEV) for _ in range(2))
        B.slkv_score(p, q, k, cu_dev, cu, own, ws, status)
        took_one = B.slkv_last_launch_count() == 1
        assert took_one or n > 735                                 # with many rows the longer ones are the general path's
        scores = own.view(hkv, n)
        assert (scores == scores[:, torch.arange(n, device=DEV) % every]).all()
        budgets = [w + 5 + 90 * h for h in range(hkv)]
        off, kept, _, _, st = both(q, k, v, cu, w, 1, budgets, domain=domain, one_launch=took_one)[0]
        for h in range(hkv):
            ref = O.select_topk(scores[h].cpu().numpy().astype(np.float64), min(n, 5 + 90 * h)).tolist()
            assert kept[int(off[h]):int(off[h + 1])].tolist() == ref + list(range(n, n + w))
        assert every > 1 or ref == list(range(len(ref)))
        cap = int(off[-1])
        out = torch.zeros(2, cap, d, device=DEV)
        B.slkv_compress(p, q, k, v, cu_dev, cu, torch.tensor(budgets, dtype=torch.int32, device=DEV), out[0], out[1],
                        torch.zeros(hkv + 1, dtype=torch.int32, device=DEV), torch.zeros(cap, dtype=torch.int32, device=DEV), ws, general, status)
        assert int(status) == 0 and int(st) == 0 and torch.equal(own, general)


@pytest.mark.parametrize("dt,d,hq,hkv,w,lens,one", [
    # layer, scores, layer with log-sum-exps handed in, scores with them
    (torch.bfloat16, 128, 32, 8, 32, [2000], (1, 1, 1, 1)), (torch.bfloat16, 128, 32, 8, 32, [8100], (1, 1, 1, 0)),
    (torch.bfloat16, 128, 32, 8, 32, [8100] * 5, (1, 0, 0, 0)), (torch.bfloat16, 64, 16, 8, 32, [8100, 100, 100, 100, 100], (0, 0, 0, 0)),
    (torch.bfloat16, 128, 32, 8, 32, [4050 + 4050 * i // 7 for i in range(8)], (0, 0, 0, 0)),
    (torch.float32, 64, 8, 8, 16, [1000], (1, 1, 1, 1)), (torch.float32, 64, 8, 8, 32, [3000], (1, 1, 1, 1)),
    (torch.float32, 128, 8, 8, 32, [3000], (1, 1, 0, 0)), (torch.float32, 128, 8, 8, 32, [4000], (0, 0, 0, 0)),
    (torch.float32, 128, 8, 8, 32, [1500, 3000], (0, 0, 0, 0)), (torch.float32, 128, 8, 8, 16, [6000], (1, 1, 1, 1)),
    (torch.float32, 64, 8, 8, 24, [2000, 4000], (1, 0, 0, 0)), (torch.float32, 128, 8, 8, 24, [2000, 4000], (0, 0, 0, 0))])
def test_what_goes_which_way(dt, d, hq, hkv, w, lens, one):
    # either side of the lines drawn for segments of unequal length, keys that do not fit at once, and calls with less to save
    q, k, v, cu = inputs(sum(lens), lens, hq, hkv, d, w, dt)
    p = B.make_params(q, k, v, w, 5, lse_units=B.SLKV_LSE_LOG2)
    cu_dev, ws = torch.tensor(cu, dtype=torch.int32, device=DEV), torch.empty(B.slkv_workspace_bytes(p, cu), dtype=torch.uint8, device=DEV)
    own, fed = (torch.zeros(B.slkv_pooled_elems(p, cu), device=DEV) for _ in range(2))
    lse, status = torch.zeros(len(lens), hq, w, device=DEV), torch.zeros(1, dtype=torch.int32, device=DEV)
    B.slkv_row_lse(p, q, k, cu_dev, cu, lse, ws)
    took = []
    for pooled, x in ((own, None), (fed, lse)):
        bud = torch.tensor([w + 40 * h for h in range(hkv)], dtype=torch.int32, device=DEV)
        res = both(q, k, v, cu, w, 5, bud.tolist(), lse=x, one_launch=False)
        same(res)
        out = torch.zeros(2, *res[0][2].shape, dtype=dt, device=DEV)
        off, kept = torch.zeros_like(res[0][0]), torch.zeros_like(res[0][1])
        B.slkv_compress(p, q, k, v, cu_dev, cu, bud, out[0], out[1], off, kept, ws, None, status, lse=x)
        took.append(B.slkv_last_launch_count() == 1)
        B.slkv_score(p, q, k, cu_dev, cu, pooled, ws, status, lse=x)
        took.append(B.slkv_last_launch_count() == 1)
    assert tuple(map(int, took)) == one and int(status) == 0 and torch.equal(own, fed)


# ---- waits that run out -------------------------------------------------------------------------------------------------
@pytest.mark.parametrize("dt,scale", [(torch.bfloat16, 1.0), (torch.bfloat16, 40.0), (torch.float32, 1.0), (torch.float32, 40.0)])
@pytest.mark.parametrize("on,supplied", [(3, False), (4, False), (4, True)])
def test_a_wait_that_runs_out_is_reported(dt, scale, on, supplied):
    # One arrival too many is expected where a segment's CTAs wait for one another: they give up after a second, the status says
    # so, whatever is written lies in the outputs, and the calls after it are right -- with scores beyond fp32's range, too, whose
    # CTAs meet twice more.
    w, hq, hkv, d, n = 16, 8, 4, 64, 1400
    q, k, v, cu = inputs(17, [n, 30, 500], hq, hkv, d, w, dt, scale)
    p = B.make_params(q, k, v, w, 7, lse_units=B.SLKV_LSE_LOG2)
    cu_dev, status = torch.tensor(cu, dtype=torch.int32, device=DEV), torch.zeros(1, dtype=torch.int32, device=DEV)
    ws = torch.empty(B.slkv_workspace_bytes(p, cu), dtype=torch.uint8, device=DEV)
    lse = None
    if supplied:
        lse = torch.zeros(3, hq, w, device=DEV)
        B.slkv_row_lse(p, q, k, cu_dev, cu, lse, ws, status)
    budgets = [40, 700, 16, 333]
    bud = torch.tensor(budgets, dtype=torch.int32, device=DEV)
    rows = sum(min(a, max(c, w)) for a in (n, 30, 500) for c in budgets)
    out = torch.full((2, rows + 64, d), 9.0, dtype=dt, device=DEV)
    off, kept = torch.zeros(3 * hkv + 1, dtype=torch.int32, device=DEV), torch.full((rows + 64,), -7, dtype=torch.int32, device=DEV)
    assert int(status) == 0
    B.slkv_debug_expire_next_wait(on)
    B.slkv_compress(p, q, k, v, cu_dev, cu, bud, out[0, :rows], out[1, :rows], off, kept[:rows], ws, None, status, lse=lse)
    assert B.slkv_last_launch_count() == 1
    torch.cuda.synchronize()
    assert int(status) == B.ERR["DEVICE_TIMEOUT"]
    assert (out[:, rows:] == 9.0).all() and (kept[rows:] == -7).all()
    a = both(q, k, v, cu, w, 7, budgets, lse=lse)
    if scale == 1.0:
        same(a)
    assert int(a[0][4]) == 0 and int(a[1][4]) == 0 and torch.equal(a[0][0], a[1][0])
