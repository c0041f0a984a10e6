"""Decode over rows cut into one to many splits, whole waves or not, against a
plain fp64 softmax; and the coarse splits of a smaller workspace."""

import pytest
import torch

from paper_2607_13205_gb300 import rolekv as R

pytestmark = pytest.mark.gpu

DEV = "cuda"


def _case(L, b, Hkv, G, d, n, lens=None, seed=0):
    g = torch.Generator(device=DEV).manual_seed(seed)
    batch = R.Batch(L, b, Hkv * G, Hkv, d, n, seqlens=lens)
    shape = (L, sum(lens), Hkv, d) if lens else (L, b, Hkv, n, d)
    k = torch.randn(shape, generator=g, device=DEV).bfloat16()
    v = torch.randn(shape, generator=g, device=DEV).bfloat16()
    q = (2 * torch.randn(L, b, Hkv * G, d, generator=g, device=DEV)).bfloat16()
    ref = torch.zeros(L, b, Hkv * G, d, dtype=torch.float64, device=DEV)
    for l in range(L):
        t0 = 0
        for s in range(b):
            m = lens[s] if lens else n
            kk, vv = (x[l, t0:t0 + m].transpose(0, 1) if lens else x[l, s] for x in (k, v))
            t0 += m if lens else 0
            if m:
                qq = q[l, s].view(Hkv, G, d).double()
                p = torch.softmax(torch.matmul(qq, kk.double().transpose(1, 2)) * d ** -0.5, -1)
                ref[l, s] = torch.matmul(p, vv.double()).view(Hkv * G, d)
    return batch, q, k, v, ref


def _run(batch, q, k, v, ws=None):
    out = torch.full(q.shape, 9.0, dtype=torch.float32, device=DEV)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    R.decode_attention(batch, q, k, v, None, 1.0, out, compacted=False, ws=ws, status=status)
    torch.cuda.synchronize()
    assert int(status) == 0
    return out


# rows: one stage and its edges, the shortest split's edges, 5 splits and more
# (merged by a CTA a head), waves that end early, packed batches
CASES = [(1, 1, 1, 1, 128, 1), (1, 1, 2, 4, 128, 64), (1, 1, 2, 4, 64, 65), (1, 1, 8, 4, 128, 128),
         (1, 1, 8, 4, 128, 129), (1, 1, 8, 7, 128, 513), (1, 1, 3, 8, 64, 641), (2, 3, 4, 4, 128, 1000),
         (1, 2, 8, 4, 128, 9001), (1, 1, 1, 5, 128, 70001), (4, 10, 8, 1, 64, 300),
         (2, 4, 4, 7, 128, 3000, (3000, 0, 1, 700)), (1, 3, 2, 2, 64, 5000, (5000, 129, 64))]


@pytest.mark.parametrize("case", CASES, ids=["x".join(map(str, c[:6])) for c in CASES])
def test_decode_splits(case):
    batch, q, k, v, ref = _case(*case)
    out = _run(batch, q, k, v)
    # fp32 logits and sums over bf16 rows: a few 2^-24 of a value's terms
    assert float((out - ref).abs().max()) < 2e-5 * max(1.0, float(ref.abs().max()))


def test_workspace_of_the_coarse_splits_is_accepted():
    batch, q, k, v, ref = _case(1, 1, 8, 4, 128, 9001)
    coarse = 8 * 9 * 4 * (128 + 2) * 4                # 9 splits of at most 1024 rows
    assert R.decode_workspace(batch, 1.0).numel() > coarse
    out = _run(batch, q, k, v, ws=torch.empty(coarse, dtype=torch.uint8, device=DEV))
    assert float((out - ref).abs().max()) < 2e-5 * max(1.0, float(ref.abs().max()))
    with pytest.raises(R.RolekvError):
        _run(batch, q, k, v, ws=torch.empty(coarse - 256, dtype=torch.uint8, device=DEV))
