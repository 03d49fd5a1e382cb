"""GPU: the list score kernel at the sizes where its walk can go wrong -- rows that fill no 32-column block, one and two
row blocks, both head dimensions, fewer tiles than CTAs, ragged last tiles, short layers sharing a group, lists that end
in mid-group -- against the oracle, and against the same layers one call at a time."""
import numpy as np
import pytest
import torch

import parity as P
from oracle import slkv_oracle as O
from paper_2508_15806_b200 import binding as B
from paper_2508_15806_b200 import synth

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


def layer(seed, lens, hq, hkv, d, w):
    g = torch.Generator().manual_seed(seed)
    T = sum(lens)
    q = torch.randn(len(lens), w, hq, d, generator=g)
    k = torch.randn(T, hkv, d, generator=g) * torch.exp(0.5 * torch.randn(T, hkv, 1, generator=g))
    return q.bfloat16(), k.bfloat16(), torch.randn(T, hkv, d, generator=g).bfloat16()


@pytest.mark.parametrize("hq,hkv,d,w", [(4, 4, 64, 5), (8, 8, 128, 16), (6, 2, 64, 16), (8, 2, 128, 33), (8, 1, 64, 31),
                                        (8, 2, 128, 64), (2, 2, 128, 129)])
@pytest.mark.parametrize("lens", [[w0 for w0 in (700,)], [130, 1, 515, 257]])
def test_rows_and_head_dims(hq, hkv, d, w, lens):
    q, k, v = layer(hq * 100 + d + w + len(lens), lens, hq, hkv, d, w)
    cu = np.concatenate([[0], np.cumsum(lens)]).tolist()
    P.check_compress(q, k, v, cu, [w + 40] * hkv, w, 5, score_path=B.SLKV_PATH_TENSOR)


@pytest.mark.parametrize("lens,n_layers,w,lse", [([300], 3, 32, False), ([4001], 19, 32, False), ([900, 33, 2000], 35, 16, True),
                                                 ([9000, 20000], 5, 64, False), ([40000], 3, 32, False)])
def test_lists_match_single_calls(lens, n_layers, w, lse):
    hq, hkv, d = 16, 4, 128
    cu = np.concatenate([[0], np.cumsum(lens)]).tolist()
    xs = [tuple(t.to(DEV) for t in layer(50 + l, lens, hq, hkv, d, w)) for l in range(n_layers)]
    p = B.make_params(*xs[0], w, 7)
    cu_dev = torch.tensor(cu, dtype=torch.int32, device=DEV)
    bud = torch.tensor([w + 30 * (h + 1) for h in range(hkv)], dtype=torch.int32, device=DEV)
    cap = sum(min(n, int(b)) for n in lens for b in bud.tolist())
    ws = torch.empty(B.slkv_workspace_bytes_overlapped(p, cu), dtype=torch.uint8, device=DEV)
    got = {}
    for fn in (B.slkv_compress, B.slkv_compress_overlapped):
        outs = []
        for q, k, v in xs:
            stats = None
            if lse:
                stats = torch.zeros(len(lens), hq, w, dtype=torch.float32, device=DEV)
                B.slkv_row_lse(p, q, k, cu_dev, cu, stats, torch.empty_like(ws))
            o = [torch.zeros(cap, d, dtype=torch.bfloat16, device=DEV), torch.zeros(cap, d, dtype=torch.bfloat16, device=DEV),
                 torch.zeros(len(lens) * hkv + 1, dtype=torch.int32, device=DEV), torch.zeros(cap, dtype=torch.int32, device=DEV),
                 torch.zeros(B.slkv_pooled_elems(p, cu), device=DEV), torch.zeros(1, dtype=torch.int32, device=DEV), stats]
            fn(p, q, k, v, cu_dev, cu, bud, *o[:4], ws, o[4], o[5], lse=stats)
            outs.append(o)
        B.slkv_join()
        torch.cuda.synchronize()
        got[fn.__name__] = outs
    for a, b in zip(*got.values()):
        assert int(a[5]) == 0 and int(b[5]) == 0
        for x, y in zip(a[:5], b[:5]):
            assert torch.equal(x, y)


@pytest.mark.parametrize("lens", [[12000], [24700], [26000, 30000, 45]])
def test_groups_of_narrow_keys(lens):
    # head_dim 64: a group is 2048 tiles of 16 KB -- layers that share one, that fill one, that are walked in several
    hq, hkv, d, w = 16, 8, 64, 16
    q, k, v = layer(70 + len(lens), lens, hq, hkv, d, w)
    cu = np.concatenate([[0], np.cumsum(lens)]).tolist()
    ref = P.oracle_pooled(q, k, cu, w, 5)
    p = B.make_params(q, k, v, w, 5)
    qd, kd, vd = (t.to(DEV) for t in (q, k, v))
    cu_dev, bud = torch.tensor(cu, dtype=torch.int32, device=DEV), torch.full((hkv,), w + 50, dtype=torch.int32, device=DEV)
    cap = sum(min(n, w + 50) for n in lens) * hkv
    ws = torch.empty(B.slkv_workspace_bytes_overlapped(p, cu), dtype=torch.uint8, device=DEV)
    outs = [[torch.zeros(*s, dtype=t, device=DEV) for s, t in (((cap, d), torch.bfloat16), ((cap, d), torch.bfloat16),
             ((len(lens) * hkv + 1,), torch.int32), ((cap,), torch.int32), ((B.slkv_pooled_elems(p, cu),), torch.float32),
             ((1,), torch.int32))] for _ in range(5)]
    for o in outs:
        B.slkv_compress_overlapped(p, qd, kd, vd, cu_dev, cu, bud, *o[:4], ws, o[4], o[5])
    B.slkv_join()
    for o in outs:
        assert int(o[5]) == 0
        P.assert_pooled_close(o[4].cpu().numpy(), ref, cu, hkv, w)


def test_scores_beyond_the_range_of_sums_without_a_reference():
    # logits of several thousand, some rows only far below zero: the rows' sums leave fp64's range
    q, k, v = layer(9, [1500], 8, 2, 128, 32)
    q, k = q * 40, k * 40
    k[:, :, 0] += 300.0
    q[:, :16, :, 0] = 80.0
    q[:, 16:, :, 0] = -80.0
    lse = P.gpu_row_lse(q, k, [0, 1500], 32)
    ref = O.row_lse(P.to_np64(q), P.to_np64(k), [0, 1500], 32, "history")
    got, ref = lse.cpu().double().numpy(), np.asarray(ref)
    assert np.all(np.isfinite(got)) and np.abs(ref).max() > 2000
    assert np.max(np.abs(got - ref) / np.abs(ref)) < 1e-5


def test_many_sequences_statistics_cleared_to_the_end():
    # 7100 sequences x 8 heads x 256 rows: the statistics area times the CTAs that clear it is more than 2^32 words.  The
    # queries overlap in memory (sequence s starts at row s), the keys are two of history and one of window per sequence.
    n, hkv, R, d = 7100, 8, 256, 64
    g = torch.Generator(device=DEV).manual_seed(5)
    rows = torch.randn(n + hkv * R, d, generator=g, device=DEV).bfloat16()
    q = rows.as_strided((n, 1, hkv * R, d), (d, hkv * R * d, d, 1))
    k = torch.randn(3 * n, hkv, d, generator=g, device=DEV).bfloat16()
    cu = list(range(0, 3 * n + 1, 3))
    p = B.make_params(q, k, None, 1, 1, score_path=B.SLKV_PATH_TENSOR)
    ws = torch.full((B.slkv_workspace_bytes(p, cu),), 0x42, dtype=torch.uint8, device=DEV)
    pooled, status = torch.zeros(n, hkv, 2, device=DEV), torch.zeros(1, dtype=torch.int32, device=DEV)
    B.slkv_score(p, q, k, torch.tensor(cu, dtype=torch.int32, device=DEV), cu, pooled, ws, status)
    assert int(status) == 0
    hist = k.view(n, 3, hkv, d)[:, :2].double()
    for a in range(0, n, 500):
        b = min(a + 500, n)
        s = torch.einsum("nhrd,njhd->nhrj", q[a:b, 0].reshape(b - a, hkv, R, d).double(), hist[a:b]) / d ** 0.5
        ref = torch.softmax(s, dim=3).mean(dim=2)
        assert torch.allclose(pooled[a:b].double(), ref, rtol=P.REL_TOL, atol=0.0), a


@pytest.mark.parametrize("hist,w,layers", [(1000, 32, 32), (32768, 32, 16), (40000, 32, 14), (65536, 64, 8)])
def test_a_list_goes_out_before_the_join(hist, w, layers):
    # layers are queued until they come to 32768 products of 128 keys x 128 rows, eight at least and thirty-two at most
    hq, hkv, d, n = 32, 8, 128, hist + w
    g = torch.Generator(device=DEV).manual_seed(hist)
    q, k = (torch.randn(*s, generator=g, device=DEV, dtype=torch.bfloat16) for s in ((1, w, hq, d), (n, hkv, d)))
    p, cu = B.make_params(q, k, k, w, 7), [0, n]
    cap = hkv * (w + 10)
    bud = torch.full((hkv,), w + 10, dtype=torch.int32, device=DEV)
    ws = torch.empty(B.slkv_workspace_bytes_overlapped(p, cu), dtype=torch.uint8, device=DEV)
    assert ws.numel() <= layers * B.slkv_workspace_bytes(p, cu)
    outs = torch.zeros(2 * layers, 2, cap, d, dtype=torch.bfloat16, device=DEV)
    off, kept = (torch.zeros(2 * layers, m, dtype=torch.int32, device=DEV) for m in (hkv + 1, cap))
    cu_dev, launches = torch.tensor(cu, dtype=torch.int32, device=DEV), []
    B.slkv_join()
    for l in range(2 * layers):
        B.slkv_compress_overlapped(p, q, k, k, cu_dev, cu, bud, outs[l, 0], outs[l, 1], off[l], kept[l], ws)
        launches.append(B.slkv_last_launch_count())
    B.slkv_join()
    torch.cuda.synchronize()
    assert launches == 2 * ([0] * (layers - 1) + [3]) and B.slkv_last_launch_count() == 0
    assert (off[:, -1] == cap).all() and torch.equal(kept, kept[:1].expand_as(kept))


@pytest.mark.parametrize("lens,n_layers,w", [([4001], 32, 32), ([2000, 33], 32, 64), ([9000, 20000], 7, 64), ([70000], 8, 32)])
def test_statistics_cleared_layer_by_layer(lens, n_layers, w):
    # layers whose statistics are cleared only after the first ones' are in use, in a workspace full of something else
    hq, hkv, d = 16, 4, 128
    cu = np.concatenate([[0], np.cumsum(lens)]).tolist()
    xs = [tuple(t.to(DEV) for t in layer(20 + l, lens, hq, hkv, d, w)) for l in range(4)]
    p = B.make_params(*xs[0], w, 7)
    cu_dev, bud = torch.tensor(cu, dtype=torch.int32, device=DEV), torch.full((hkv,), w + 30, dtype=torch.int32, device=DEV)
    cap, n = sum(min(x, w + 30) for x in lens) * hkv, B.slkv_workspace_bytes_overlapped(p, cu)
    ws = torch.empty(n, dtype=torch.uint8, device=DEV)
    kv, off, kept = torch.zeros(2, cap, d, dtype=torch.bfloat16, device=DEV), torch.zeros(len(lens) * hkv + 1, dtype=torch.int32, device=DEV), torch.zeros(cap, dtype=torch.int32, device=DEV)
    scores, status = torch.zeros(4 + 2 * n_layers, B.slkv_pooled_elems(p, cu), device=DEV), torch.zeros(1, dtype=torch.int32, device=DEV)
    for l, x in enumerate(xs):
        B.slkv_compress(p, *x, cu_dev, cu, bud, *kv, off, kept, ws, scores[l], status)
    for turn in range(2):
        ws.fill_(0x42)
        for l in range(n_layers):
            B.slkv_compress_overlapped(p, *xs[l % 4], cu_dev, cu, bud, *kv, off, kept, ws, scores[4 + turn * n_layers + l], status)
        B.slkv_join()
    assert int(status) == 0
    for l in range(2 * n_layers):
        assert torch.equal(scores[4 + l], scores[l % n_layers % 4])
