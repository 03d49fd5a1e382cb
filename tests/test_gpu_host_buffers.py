"""GPU: slkv_compress_host with page-locked and pageable buffers in every role, against the device entry point."""
import itertools

import numpy as np
import pytest
import torch

import parity as P
from paper_2508_15806_b200 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lens,dt,d", [([700, 3, 90], torch.bfloat16, 128), ([257], torch.float32, 64), ([10] * 70, torch.float32, 64)])
def test_buffers(lens, dt, d):
    w, hq, hkv = 8, 4, 2
    g = torch.Generator().manual_seed(len(lens))
    T = sum(lens)
    q, k, v = (torch.randn(len(lens), w, hq, d, generator=g).to(dt), torch.randn(T, hkv, d, generator=g).to(dt),
               torch.randn(T, hkv, d, generator=g).to(dt))
    cu, bud = np.concatenate([[0], np.cumsum(lens)]).tolist(), [40, 1]
    ref = P.gpu_compress(q, k, v, cu, bud, w, 5)
    n = int(ref["offsets"][-1])
    p = B.make_params(q, k, v, w, 5)
    arena = torch.empty(B.slkv_compress_host_arena_bytes(p, cu, n + 5), dtype=torch.uint8, device="cuda:0")
    for pin_in, pin_rows, pin_idx in itertools.product((True, False), repeat=3):
        f = lambda t, on: t.pin_memory() if on else t.clone()                                      # noqa: E731
        ko, vo = (f(torch.full((n + 5, d), 7, dtype=dt), pin_rows) for _ in range(2))
        off, kept = f(torch.zeros(len(lens) * hkv + 1, dtype=torch.int32), pin_idx), f(torch.full((n + 5,), -9, dtype=torch.int32), pin_idx)
        rows = B.slkv_compress_host(p, f(q, pin_in), f(k, pin_in), f(v, pin_in), cu, torch.tensor(bud, dtype=torch.int32), ko, vo,
                                    off, kept, arena)
        assert rows == n and off.tolist() == ref["offsets"].tolist()
        assert kept[:n].tolist() == ref["kept_idx"][:n].tolist() and (kept[n:] == -9).all()
        assert torch.equal(ko[:n], ref["k_out"][:n]) and torch.equal(vo[:n], ref["v_out"][:n]) and (vo[n:] == 7).all()
