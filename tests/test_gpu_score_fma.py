"""GPU: the fp32 FMA score kernel at the edges of its tiles (64 keys x 64 rows), with rows that do not fit in shared memory
at once, and with scores whose sums leave fp32's range, against the oracle."""
import numpy as np
import pytest
import torch

import parity as P
from oracle import slkv_oracle as O
from paper_2508_15806_b200 import binding as B

pytestmark = pytest.mark.gpu


def layer(seed, lens, hq, hkv, d, w, dt):
    g = torch.Generator().manual_seed(seed)
    T = sum(lens)
    return (torch.randn(len(lens), w, hq, d, generator=g).to(dt), torch.randn(T, hkv, d, generator=g).to(dt),
            torch.randn(T, hkv, d, generator=g).to(dt))


@pytest.mark.parametrize("hq,hkv,d,w,dt", [(2, 2, 64, 1, torch.float32), (6, 2, 64, 21, torch.float32), (4, 1, 128, 17, torch.float32),
                                           (8, 1, 128, 100, torch.float32), (5, 5, 64, 64, torch.bfloat16), (4, 2, 128, 65, torch.bfloat16)])
@pytest.mark.parametrize("extra", [[1, 63, 64, 65, 128, 129], [700, 0, 2000]])
@pytest.mark.parametrize("domain", [B.SLKV_HISTORY, B.SLKV_ALL_CAUSAL])
def test_tile_edges(hq, hkv, d, w, dt, extra, domain):
    lens = [w + e for e in extra]
    q, k, v = layer(hq + d + w + len(extra), lens, hq, hkv, d, w, dt)
    cu = np.concatenate([[0], np.cumsum(lens)]).tolist()
    P.check_compress(q, k, v, cu, [w + 20] * hkv, w, 3, score_path=B.SLKV_PATH_SIMT, domain=domain)


@pytest.mark.parametrize("d", [64, 128])
def test_sums_beyond_fp32(d):
    q, k, _ = layer(3, [900], 4, 2, d, 8, torch.float32)
    k[:, :, 0] += 60.0
    q[:, :4, :, 0], q[:, 4:, :, 0] = 70.0, -70.0
    lse = P.gpu_row_lse(q, k, [0, 900], 8, score_path=B.SLKV_PATH_SIMT).cpu().double().numpy()
    ref = np.asarray(O.row_lse(P.to_np64(q), P.to_np64(k), [0, 900], 8, "history"))
    assert np.abs(ref).max() > 200 and np.max(np.abs(lse - ref) / np.abs(ref)) < 1e-5


def test_many_sequences_statistics_cleared_to_the_end():
    # 52430 sequences x 8 heads x 1024 rows: the statistics area is more than 2^31 words.  One history key per sequence
    # takes every row's whole weight.  The queries overlap in memory (sequence s starts at row s).
    n, hkv, R, d = 52430, 8, 1024, 64
    dev = torch.device("cuda:0")
    g = torch.Generator(device=dev).manual_seed(6)
    q = torch.randn(n + hkv * R, d, generator=g, device=dev).as_strided((n, 1, hkv * R, d), (d, hkv * R * d, d, 1))
    k = torch.randn(2 * n, hkv, d, generator=g, device=dev)
    cu = list(range(0, 2 * n + 1, 2))
    p = B.make_params(q, k, None, 1, 1, score_path=B.SLKV_PATH_SIMT)
    ws = torch.full((B.slkv_workspace_bytes(p, cu),), 0x42, dtype=torch.uint8, device=dev)
    pooled, status = torch.zeros(n * hkv, device=dev), torch.zeros(1, dtype=torch.int32, device=dev)
    B.slkv_score(p, q, k, torch.tensor(cu, dtype=torch.int32, device=dev), cu, pooled, ws, status)
    assert int(status) == 0
    assert torch.allclose(pooled, torch.ones_like(pooled), rtol=P.REL_TOL, atol=0.0)
