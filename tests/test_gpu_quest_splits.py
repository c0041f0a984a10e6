"""Quest bounds with a unit's pages on one to many CTAs: row lengths around
page and CTA edges, few and many units, against the bound in fp64."""

import pytest
import torch

from paper_2607_13205_gb300 import rolekv as R

pytestmark = pytest.mark.gpu

DEV = "cuda"


def _bounds(k, qbar, page):
    """k [H][n][d], qbar [H][d] -> [H][n]"""
    out = torch.empty(k.shape[:2], dtype=torch.float64, device=DEV)
    for t in range(0, k.shape[1], page):
        x = k[:, t:t + page].double()
        out[:, t:t + page] = torch.maximum(qbar * x.amin(1), qbar * x.amax(1)).sum(-1)[:, None]
    return out


CASES = [(1, 1, 1, 1, 128, 1, 16, 8), (1, 1, 2, 4, 64, 17, 16, 8), (1, 1, 8, 4, 128, 4095, 16, 64),
         (1, 1, 8, 4, 128, 4097, 8, 32), (1, 1, 1, 7, 128, 40000, 64, 32), (60, 1, 8, 1, 64, 33, 16, 8),
         (2, 4, 4, 7, 128, 3000, 16, 32, (3000, 0, 1, 700)), (1, 2, 4, 8, 128, 257, 4096, 32),
         (1, 1, 1, 4, 128, 20001, 2, 64, (20001,)), (2, 3, 2, 4, 64, 9001, 8, 32, (9001, 7, 4000))]


@pytest.mark.parametrize("case", CASES, ids=["x".join(map(str, c[:8])) for c in CASES])
def test_quest_page_splits(case):
    L, b, Hkv, G, d, n, page, W = case[:8]
    lens = case[8] if len(case) > 8 else None
    g = torch.Generator(device=DEV).manual_seed(5)
    batch = R.Batch(L, b, Hkv * G, Hkv, d, n, seqlens=lens)
    k = torch.randn((L, sum(lens), Hkv, d) if lens else (L, b, Hkv, n, d), generator=g, device=DEV).bfloat16()
    q = torch.randn(L, b, Hkv * G, W, d, generator=g, device=DEV).bfloat16()
    sc = torch.full(batch.score_shape(), -9.0, device=DEV)
    R.quest_score(batch, q, k, W, page, sc)
    torch.cuda.synchronize()
    for l in range(L):
        t0 = 0
        for s in range(b):
            m = lens[s] if lens else n
            kk = k[l, t0:t0 + m].transpose(0, 1) if lens else k[l, s]
            got = sc[l, :, t0:t0 + m] if lens else sc[l, s]
            t0 += m if lens else 0
            if m == 0:
                continue
            qbar = q[l, s].view(Hkv, G, W, d)[:, :, :min(W, m)].double().mean((1, 2))
            ref = _bounds(kk, qbar, page)
            # fp32 sums of d products of order one
            assert float((got - ref).abs().max()) < 1e-5 * max(1.0, float(ref.abs().max()))
