"""Packed batches whose CTAs take items without key tiles (an empty sequence,
or a chunk of a short one) between items of a tile or two: each item uses its
own normalisers, in two passes and with supplied ones."""

import pytest
import torch

from paper_2607_13205_gb300 import inputs as I
from paper_2607_13205_gb300 import rolekv as R
from tests.gpu_helpers import SCORE_RTOL, lib_batch

pytestmark = pytest.mark.gpu

DEV = "cuda"

# (L, Hkv, G, d, sequence lengths).  With 152 CTAs a CTA's items are 152 apart:
CASES = {
    # one chunk a unit; sequences 0, 2, 1, 0 of a CTA: empty, then one tile
    "empty_then_one_tile": (40, 4, 4, 128, (0, 2000, 100)),
    # sequences 0, 3, 1, 4, 2: two empty ones, one tile, empty again
    "empty_runs": (50, 4, 2, 64, (0, 100, 2000, 0, 1)),
    # four chunks a unit; sequences 0, 1, 2: the last chunk has 63 tiles of 250,
    # none of 9 and one of 13
    "last_chunk": (20, 2, 4, 128, (32000, 1100, 1600)),
    # two chunks a unit, the second without tiles up to 128 tokens, with one up to 384
    "second_chunk": (40, 4, 7, 128, (8300, 128, 300)),
}


@pytest.mark.parametrize("name", CASES)
def test_items_without_tiles(name):
    L, Hkv, G, d, lens = CASES[name]
    w = I.Workload("gap", "snapkv", L, len(lens), Hkv * G, Hkv, d, max(lens), 32, 1, (0.1,), 4, (3, 5), (1, 3),
                   seqlens=lens)
    K, _ = I.make_kv(w, I.workload_roles(w, 5), 5, device=DEV, with_v=False)
    qw = I.make_q_window(w, 5, device=DEV)
    lse = torch.zeros(L, w.b, w.Hq, w.W, device=DEV)
    ref = torch.zeros(L, Hkv, sum(lens), dtype=torch.float64, device=DEV)
    t0 = 0
    for s, n in enumerate(lens):
        if n:
            we = min(w.W, n)
            pos = torch.arange(n - we, n, device=DEV).repeat(G)
            late = torch.arange(n, device=DEV)[None, :] > pos[:, None]
            for l in range(L):
                q = qw[l, s].double().view(Hkv, G, w.W, d)[:, :, :we].reshape(Hkv, G * we, d)
                x = torch.matmul(q, K[l, t0:t0 + n].double().permute(1, 2, 0)) * d ** -0.5
                x.masked_fill_(late, float("-inf"))
                lse[l, s, :, :we] = torch.logsumexp(x, dim=-1).view(w.Hq, we).float()
                ref[l, :, t0:t0 + n] = torch.softmax(x, dim=-1).sum(-2)
        t0 += n
    batch = lib_batch(w, DEV)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    for given in (None, lse):
        for _ in range(8):
            sc = torch.empty(batch.score_shape(), device=DEV)
            R.snapkv_score(batch, qw, K, w.W, 1, sc, lse_win=given, status=status)
            assert int(status) == 0
            assert float(((sc - ref).abs() / ref).max()) < SCORE_RTOL
