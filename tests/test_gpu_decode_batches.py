"""A decode step's outputs do not depend on what else is in the batch beyond
fp32 rounding: where a unit's rows are cut follows the whole batch and the
workspace, so the last bits may differ, and each stays as close to the exact
result."""

import pytest
import torch

from paper_2607_13205_gb300 import rolekv as R

pytestmark = pytest.mark.gpu

DEV = "cuda"

# Sums of m products of probabilities (adding to 1) and values of order one in
# fp32, from logits of order 4 with an error of d roundings: the output's error
# is a few times 2^-24 of the largest value.
BOUND = 2e-6


@pytest.mark.parametrize("d,G,b,m", [(128, 4, 4, 3277), (64, 8, 3, 820), (128, 7, 1, 20000), (64, 1, 2, 65)])
def test_layers_one_at_a_time_and_a_small_workspace(d, G, b, m):
    L, Hkv = 24, 4
    g = torch.Generator(device=DEV).manual_seed(3)
    k = torch.randn(L, b, Hkv, m, d, generator=g, device=DEV).bfloat16()
    v = torch.randn(L, b, Hkv, m, d, generator=g, device=DEV).bfloat16()
    q = torch.randn(L, b, Hkv * G, d, generator=g, device=DEV).bfloat16()
    whole, layer = R.Batch(L, b, Hkv * G, Hkv, d, m), R.Batch(1, b, Hkv * G, Hkv, d, m)

    def run(batch, l, n, ws=None):
        out = torch.empty((n, b, Hkv * G, d), device=DEV)
        return R.decode_attention(batch, q[l:l + n], k[l:l + n], v[l:l + n], None, 1.0, out, compacted=False, ws=ws)

    x = torch.matmul(q.double().view(L, b, Hkv, G, d), k.double().transpose(-1, -2)) * d ** -0.5
    ref = torch.matmul(torch.softmax(x, dim=-1), v.double()).view(L, b, Hkv * G, d)
    coarse = L * b * Hkv * -(-m // 1024) * G * (d + 2) * 4
    assert coarse <= R.decode_workspace(whole, 1.0).numel()
    outs = [run(whole, 0, L), torch.cat([run(layer, l, 1) for l in range(L)]),
            run(whole, 0, L, torch.empty(coarse, dtype=torch.uint8, device=DEV))]
    for o in outs:
        assert float((o - ref).abs().max()) < BOUND * float(v.abs().max())
    # the same batch and workspace: the same bits
    assert torch.equal(outs[0], run(whole, 0, L))
