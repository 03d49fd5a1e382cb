"""GPU: lists whose pooled scores nobody asks for take one product with every key and exact votes for the keys that may be kept
(slkv_bound.cu); the same list with pooled scores takes the votes of all keys.  What is kept is the same bit for bit, whatever the
sizes, strides, budgets and values: estimates that bound nothing, ties, scores beyond fp32's range, values that are not finite."""
import numpy as np
import pytest
import torch

from paper_2508_15806_b200 import binding as B
import parity as P

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


@pytest.fixture(autouse=True)
def hooks_off():
    yield
    B.slkv_debug_list_way(0)
    B.slkv_debug_expire_next_wait(0)
    B.slkv_profile_enable(0)
    B.slkv_profile_collect()


LONG = 66000            # a sequence whose segments are a cluster's


def inputs(kind, seed, lens, hq, hkv, d, w):
    g = torch.Generator(device=DEV).manual_seed(seed)
    T, n, G = sum(lens), len(lens), hq // hkv
    q = torch.randn(n, w, hq, d, generator=g, device=DEV)
    k = torch.randn(T, hkv, d, generator=g, device=DEV)
    v = torch.randn(T, hkv, d, generator=g, device=DEV).bfloat16()
    if kind == "stripes":                                # keys that all rows look at, and some rows' own
        u = torch.randn(1, hkv, d, generator=g, device=DEV)
        u = u / u.norm(dim=2, keepdim=True)
        q = q + 4.0 * u.repeat_interleave(G, dim=1)
        amp = 1.5 * torch.randn(T, hkv, 1, generator=g, device=DEV)
        amp[torch.randint(0, T, (1 + T // 500,), generator=g, device=DEV)] += 8.0
        k = k + amp * u * (d ** 0.5 / 4.0)
    elif kind == "ties":                                 # a few different keys, and many of each
        k = k[torch.randint(0, 5, (T,), generator=g, device=DEV)]
    elif kind == "same":
        k = k[:1].expand(T, hkv, d).clone()
    elif kind == "late":                                 # the rows' mass lies in one key, behind all samples, a key for each row
        k[T - w - 3] *= 6.0
        k[T // 2] *= 8.0
    elif kind == "large":                                # scores of +- 1000 and more
        q, k = 30.0 * q, 10.0 * k
    elif kind == "small":                                # every score near -200: sums below fp32's range
        q = torch.ones_like(q) + 0.01 * q
        k = -200.0 / d ** 0.5 + 0.3 * k
    elif kind == "cancel":                               # small differences of large products
        q[..., ::2] += 40.0
        q[..., 1::2] -= 40.0
        k[..., ::2] += 20.0
        k[..., 1::2] += 20.0
    elif kind == "not finite":
        k[T // 3, 0, 0] = float("inf")
        k[T // 5, hkv - 1, 1] = float("nan")
        q[0, 0, 0, 0] = float("nan")
    return q.bfloat16(), k.bfloat16(), v


def one_list(layers, lens, w, pool, budgets, way, pooled=False, room=None, **kw):
    """The layers' outputs (k, v, offsets, kept positions, status), and the score kernel they took."""
    cu = np.concatenate([[0], np.cumsum(lens)]).tolist()
    p = B.make_params(*layers[0], w, pool, **kw)
    hkv, d = layers[0][1].shape[1:]
    cu_dev = torch.tensor(cu, dtype=torch.int32, device=DEV)
    ws = torch.full((B.slkv_workspace_bytes_overlapped(p, cu),), 0x5a, dtype=torch.uint8, device=DEV)
    outs = []
    B.slkv_debug_list_way(way)
    B.slkv_profile_enable(2)
    for (q, k, v), bud in zip(layers, budgets):
        cap = room or sum(min(n, max(int(b), w)) for n in lens for b in bud)
        b = torch.tensor(bud, dtype=torch.int32, device=DEV)
        o = [torch.full((cap, d), 7, dtype=torch.bfloat16, device=DEV), torch.full((cap, d), 7, dtype=torch.bfloat16, device=DEV),
             torch.zeros(len(lens) * hkv + 1, dtype=torch.int32, device=DEV), torch.full((cap,), -1, dtype=torch.int32, device=DEV),
             torch.zeros(1, dtype=torch.int32, device=DEV)]
        scores = torch.zeros(B.slkv_pooled_elems(p, cu), device=DEV) if pooled else None
        B.slkv_compress_overlapped(p, q, k, v, cu_dev, cu, b, *o[:4], ws, scores, o[4])
        outs.append(o + [b, scores])                     # the calls are queued: what they use stays
    B.slkv_join()
    torch.cuda.synchronize()
    B.slkv_profile_enable(0)
    B.slkv_debug_list_way(0)
    return outs, set(B.slkv_profile_collect())


def both_ways(layers, lens, w, pool, budgets, **kw):
    """The list without and with pooled scores."""
    got = []
    for pooled in (False, True):
        outs, kernels = one_list(layers, lens, w, pool, budgets, 1, pooled, **kw)
        assert kernels == {"k_score_list" if pooled else "k_score_bound"}
        got.append(outs)
    for one, all_votes in zip(*got):
        assert int(one[4]) == 0 and int(all_votes[4]) == 0
        assert torch.equal(one[2], all_votes[2])
        assert torch.equal(one[3], all_votes[3])
        for i in (0, 1):
            assert torch.equal(one[i].view(torch.int16), all_votes[i].view(torch.int16))


KINDS = ["gaussian", "stripes", "ties", "same", "late", "large", "small", "cancel", "not finite"]


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("hq,hkv,d,w,lens", [(8, 2, 128, 32, [4000, LONG]), (8, 4, 64, 64, [700, 33, 2500, 2 * LONG]), (16, 2, 128, 20, [33001]),
                                             (8, 1, 64, 31, [LONG, 300])])
def test_what_is_kept_is_what_all_votes_keep(kind, hq, hkv, d, w, lens):
    layers = [inputs(kind, 31 * l + w, lens, hq, hkv, d, w) for l in range(3)]
    budgets = [[w + x for x in (0, 1, 9, 100)][:hkv] if hkv > 2 else [w + 3 ** (l + 2), w + 11 * (l + 1)][:hkv] for l in range(3)]
    both_ways(layers, lens, w, 7, budgets)


@pytest.mark.parametrize("hq,hkv,d,w", [(3, 1, 128, 22), (8, 1, 64, 9), (2, 1, 64, 64), (8, 2, 128, 33), (3, 1, 128, 85), (8, 2, 128, 64)])
@pytest.mark.parametrize("n", [1, 15, 16, 127, 128, 129, 2047, 2049, 4097, 8195, 16390])
def test_rows_and_tile_edges(hq, hkv, d, w, n):
    layers = [inputs("stripes", n + l, [LONG, n + w], hq, hkv, d, w) for l in range(2)]
    both_ways(layers, [LONG, n + w], w, 5, [[w + max(1, n // 40)] * hkv, [w + 1] * hkv])


@pytest.mark.parametrize("pool", [1, 3, 5, 9])
@pytest.mark.parametrize("share", [0.0, 0.001, 0.0158, 0.016, 0.1, 0.3, 0.97, 1.0])
def test_budgets_around_the_line_to_all_votes(pool, share):
    w, n, hkv = 32, 32100, 4
    layers = [inputs("stripes", l, [n + w], 16, hkv, 128, w) for l in range(3)]
    k = int(share * n)
    both_ways(layers, [n + w], w, pool, [[w + k, w + 20, w + k + 1, w - 5], [w + 7] * 4, [w + k] * 4])


def test_all_causal_domain_and_strides():
    w, n, hq, hkv, d = 24, 33003, 8, 2, 128
    layers = []
    for l in range(3):
        q, k, v = inputs("stripes", l, [n + w], hq, hkv, d, w)
        fused = torch.cat([k, v], dim=1).contiguous()              # K and V slices of one buffer, heads outside tokens for q
        layers.append((q.permute(0, 2, 1, 3).contiguous().permute(0, 2, 1, 3), fused[:, :hkv], fused[:, hkv:]))
    both_ways(layers, [n + w], w, 7, [[w + 60, w + 5]] * 3, softmax_domain=B.SLKV_ALL_CAUSAL)


@pytest.mark.parametrize("lens,w", [([131072], 64), ([40000, 100, 262000], 17)])
def test_segments_of_several_ctas(lens, w):
    layers = [inputs("stripes", l, lens, 8, 2, 128, w) for l in range(2)]
    both_ways(layers, lens, w, 7, [[w + 300, w + 2], [w + 1500, w + 9000]])


@pytest.mark.parametrize("n", [33000, 66000])           # a CTA per segment, a cluster
@pytest.mark.parametrize("stripe,rest", [(-59, -90), (-53, -90), (-47, -90), (-53, -74), (-47, -66)])
def test_keys_whose_exponentials_are_below_fp32(n, stripe, rest):
    """Rows whose every score is so low that a key's exponential is zero in fp32 though its share of the row is not (2^-126 and
    2^-75 and the like), and one row that makes the threshold lower still.  Queries along two axes: scores of 1.02 k (log2)."""
    w, hq, hkv, d = 32, 8, 2, 128
    q, k = torch.zeros(1, w, hq, d, device=DEV), torch.zeros(n + w, hkv, d, device=DEV)
    q[..., 0] = 8.0
    q[0, 5, 1, 0], q[0, 5, 1, 1] = 0.0, 8.0                       # one row of the first segment looks along the other axis
    k[..., 0], k[..., 1] = -137.0, rest
    k[::128, :, 0], k[::128, :, 1] = stripe, stripe + 2
    k[n // 3 + 5, :, 1] = -10.0
    low = 2 * n // 3 + 9
    k[low, :, 0], k[low, :, 1] = -124.0, -137.0
    v = torch.randn(n + w, hkv, d, device=DEV).bfloat16()
    k = k.bfloat16()
    keep = n // 128 + 44
    both_ways([(q.bfloat16(), k, v)] * 2, [n + w], w, 1, [[w + keep, w + 3], [w + 5, w + keep]])


@pytest.mark.parametrize("n,hkv", [(40001, 4), (70003, 2), (131000, 2), (262002, 1)])          # clusters of 2, 4, 4 and 8
def test_borders_between_the_ctas_of_a_cluster_in_a_second_round(n, hkv):
    """The weightiest key is one that few CTAs saw when they weighed their rows: thresholds come out too high, and are taken again
    from the votes.  Around every border between slices lie keys on either side of the line."""
    w, d, hq = 32, 128, 4 * hkv
    layers = []
    for l in range(2):
        q, k, v = inputs("stripes", 7 * l + n % 5, [n + w], hq, hkv, d, w)
        g = torch.Generator(device=DEV).manual_seed(n + l)
        u = q[0, 0, ::4].float()
        u = u / u.norm(dim=1, keepdim=True)
        cs = 2
        while (n + 3 + cs - 1) // cs + 3 > 32768:
            cs *= 2
        for h in range(hkv):
            shift = h * n & 3
            slice_ = ((n + shift + cs - 1) // cs + 3) & ~3
            for rank in range(1, cs):
                p = rank * slice_ - shift + torch.arange(-6, 6, device=DEV)
                amp = 4.0 + 4.0 * torch.rand(12, 1, generator=g, device=DEV)
                k[p, h] = (0.3 * torch.randn(12, d, generator=g, device=DEV) + amp * u[h] * (d ** 0.5 / 4.0)).bfloat16()
            k[n // 2 + 11, h] = (16.0 * u[h] * (d ** 0.5 / 4.0)).bfloat16()
        layers.append((q, k, v))
    for pool in (3, 7):
        both_ways(layers, [n + w], w, pool, [[w + 40 + 90 * h for h in range(hkv)], [w + 400 - 30 * h for h in range(hkv)]])


@pytest.mark.parametrize("rows", ["one row", "a segment", "all"])
@pytest.mark.parametrize("n", [33001, 66003])
def test_votes_that_are_not_finite(rows, n):
    """Query rows that are not finite: every vote of the segment is not, and the edges decide what is kept."""
    w, hq, hkv, d = 32, 8, 2, 128
    layers = [inputs("stripes", l, [n + w, 700], hq, hkv, d, w) for l in range(2)]
    for q, _, _ in layers:
        if rows == "one row":
            q[0, w - 1, hq - 1, 0] = float("nan")
        elif rows == "a segment":
            q[0, :, :hq // hkv, 3] = float("nan")
        else:
            q[:] = float("inf")
    both_ways(layers, [n + w, 700], w, 7, [[w + 60, w + 5], [w + 3, w + 2000]])


@pytest.mark.parametrize("hq,hkv,d,w,lens", [(16, 4, 128, 32, [LONG, 9000, 40, 33000, 1300, 20000, 128 + 32, 60001]), (16, 16, 64, 80, [LONG]),
                                             (32, 8, 128, 32, [17000] * 3), (8, 2, 128, 64, [2 * LONG, 700]), (6, 1, 64, 40, [200000, 513 + 40])])
@pytest.mark.parametrize("share", [0.1, 0.5, 0.9])
def test_heads_that_need_all_votes_among_others(hq, hkv, d, w, lens, share):
    """Any mixture of heads that keep few positions and many, in all layers and of sequences of any length."""
    rng = np.random.default_rng(len(lens) * hq + int(10 * share))
    n_layers = 8 if sum(lens) < 70000 else 5
    layers = [inputs("stripes", l + w, lens, hq, hkv, d, w) for l in range(n_layers)]
    budgets = [[int(w + (rng.integers(600, 6000) if rng.random() < share else rng.integers(0, 400))) for _ in range(hkv)] for _ in layers]
    both_ways(layers, lens, w, 7, budgets)


@pytest.mark.parametrize("n", [16300, 32764, 32800])        # 16 and 32 positions a thread, a cluster
def test_against_the_oracle(n):
    w, hq, hkv, d = 32, 8, 2, 128
    lens = [n + w, 9000]
    layers = [inputs(kind, n + l, lens, hq, hkv, d, w) for l, kind in enumerate(["stripes", "gaussian"])]
    budgets = [[w + 100, w + 400], [w + 10, w + 700]]
    outs, kernels = one_list(layers, lens, w, 7, budgets, 1)
    assert kernels == {"k_score_bound"}
    cu = [0, lens[0], sum(lens)]
    for (q, k, v), o, bud in zip(layers, outs, budgets):
        gpu = {"offsets": o[2].cpu().numpy().astype(np.int64), "kept_idx": o[3].cpu().numpy().astype(np.int64), "k_out": o[0].cpu(), "v_out": o[1].cpu()}
        assert int(o[4]) == 0
        P.assert_selection_valid(gpu, P.oracle_pooled(q.cpu(), k.cpu(), cu, w, 7), cu, bud, w, k.cpu(), v.cpu())


@pytest.mark.parametrize("n_layers,keep,room,pooled,kernel", [
    (31, 100, None, False, "k_score_bound"), (31, 100, None, True, "k_score_list"), (31, 100, 8 * 17000, False, "k_score_bound"),
    (31, 512, None, False, "k_score_list"), (18, 20, None, False, "k_score_bound"), (18, 400, None, False, "k_score_list"),
    (8, 20, None, False, "k_score_list")])
def test_which_way_a_list_goes(n_layers, keep, room, pooled, kernel):
    """17000 tokens, 8 KV heads, 128 rows: 1064 products a layer.  Few of them, or much to keep, and two products are quicker; room
    for every row tells nothing of what is kept."""
    w = 32
    x = inputs("gaussian", 1, [17000], 32, 8, 128, w)
    _, kernels = one_list([x] * n_layers, [17000], w, 7, [[w + keep] * 8] * n_layers, 0, pooled, room)
    assert kernels == {kernel}


@pytest.mark.parametrize("wait", [1, 2])                     # for the statistics, for their clearing
def test_a_wait_that_runs_out(wait):
    """Every CTA gives up after its limit, the status words say so, and the next list is right."""
    w, lens = 32, [33032]
    layers = [inputs("stripes", l, lens, 8, 2, 128, w) for l in range(3)]
    budgets = [[w + 50, w + 900]] * 3                        # the second head gets all its votes: those wait for the statistics
    B.slkv_debug_expire_next_wait(wait)
    outs, kernels = one_list(layers, lens, w, 7, budgets, 1)
    assert kernels == {"k_score_bound"}
    assert all(int(o[4]) == B.ERR["DEVICE_TIMEOUT"] for o in outs)
    both_ways(layers, lens, w, 7, budgets)
