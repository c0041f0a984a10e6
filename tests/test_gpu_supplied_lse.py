"""Scores with supplied normalisers on batches whose CTAs take several items in
a row: an item's normalisers and positions must not replace the ones other
warps still read.  (They did: a few tiles at the causal edge came out wrong in
some runs.)"""

import pytest
import torch

from paper_2607_13205_gb300 import inputs as I
from paper_2607_13205_gb300 import rolekv as R
from tests.gpu_helpers import SCORE_RTOL, lib_batch

pytestmark = pytest.mark.gpu

DEV = "cuda"


def _logits(q, k, pos0):
    x = torch.matmul(q.double(), k.double().T) * q.shape[-1] ** -0.5
    row = torch.arange(pos0, pos0 + q.shape[0], device=DEV)
    return x.masked_fill_(torch.arange(k.shape[0], device=DEV)[None, :] > row[:, None], float("-inf"))


@pytest.mark.parametrize("shape", [(5, 1, 2, 5, 128, 2133), (2, 3, 2, 5, 128, 1500), (1, 1, 8, 4, 64, 4001)])
def test_h2o_with_lse_many_items_a_cta(shape):
    L, b, Hkv, G, d, n = shape
    w = I.Workload("lse", "h2o", L, b, Hkv * G, Hkv, d, n, 8, 1, (0.1,), 4, (3, 5), (1, 3))
    K, _ = I.make_kv(w, I.workload_roles(w, 2), 2, device=DEV, with_v=False)
    Q = I.make_q_full(w, 2, device=DEV)
    lse = torch.empty(L, b, w.Hq, n, device=DEV)
    ref = torch.zeros(L, b, Hkv, n, dtype=torch.float64, device=DEV)
    for l in range(L):
        for s in range(b):
            for h in range(w.Hq):
                x = _logits(Q[l, s, h], K[l, s, h // G], 0)
                lse[l, s, h] = torch.logsumexp(x, dim=-1)
                ref[l, s, h // G] += torch.softmax(x, dim=-1).sum(0)
    batch = lib_batch(w, DEV)
    for _ in range(8):
        sc = torch.empty(batch.score_shape(), device=DEV)
        R.h2o_score(batch, Q, K, sc, lse=lse)
        assert float(((sc - ref).abs() / ref).max()) < SCORE_RTOL


def test_window_lse_many_items_a_cta():
    w = I.Workload("lse", "snapkv", 16, 2, 56, 8, 128, 1100, 32, 1, (0.1,), 4, (3, 5), (1, 3))
    K, _ = I.make_kv(w, I.workload_roles(w, 2), 2, device=DEV, with_v=False)
    qw = I.make_q_window(w, 2, device=DEV)
    q = qw.double().view(w.L, w.b, w.Hkv, w.G * w.W, w.d)
    x = torch.matmul(q, K.double().transpose(-1, -2)) * w.d ** -0.5
    pos = torch.arange(w.n - w.W, w.n, device=DEV).repeat(w.G)
    x.masked_fill_(torch.arange(w.n, device=DEV)[None, :] > pos[:, None], float("-inf"))
    lse = torch.logsumexp(x, dim=-1).view(w.L, w.b, w.Hq, w.W).float()
    ref = torch.softmax(x, dim=-1).sum(-2)
    batch = lib_batch(w, DEV)
    for _ in range(8):
        sc = torch.empty(batch.score_shape(), device=DEV)
        R.snapkv_score(batch, qw, K, w.W, 1, sc, lse_win=lse)
        assert float(((sc - ref).abs() / ref).max()) < SCORE_RTOL


def test_window_lse_with_empty_sequences():
    """Empty items between full ones: the tensor core's warp must not take an
    empty item's normaliser barrier for the next one's."""
    lens = (700, 0, 0, 1, 0, 513, 0, 0, 0, 1100, 0, 300) * 4
    w = I.Workload("lse", "snapkv", 6, len(lens), 8, 2, 128, max(lens), 32, 1, (0.1,), 4, (3, 5), (1, 3), seqlens=lens)
    K, _ = I.make_kv(w, I.workload_roles(w, 3), 3, device=DEV, with_v=False)
    qw = I.make_q_window(w, 3, device=DEV)
    lse = torch.zeros(w.L, w.b, w.Hq, w.W, device=DEV)
    ref = torch.zeros(w.L, w.Hkv, sum(lens), dtype=torch.float64, device=DEV)
    t0 = 0
    for s, n in enumerate(lens):
        if n:
            we = min(w.W, n)
            q = qw[:, s].double().view(w.L, w.Hkv, w.G, w.W, w.d)[:, :, :, :we].reshape(w.L, w.Hkv, w.G * we, w.d)
            x = torch.matmul(q, K[:, t0:t0 + n].double().permute(0, 2, 3, 1)) * w.d ** -0.5
            pos = torch.arange(n - we, n, device=DEV).repeat(w.G)
            x.masked_fill_(torch.arange(n, device=DEV)[None, :] > pos[:, None], float("-inf"))
            lse[:, s, :, :we] = torch.logsumexp(x, dim=-1).view(w.L, w.Hq, we).float()
            ref[:, :, t0:t0 + n] = torch.softmax(x, dim=-1).sum(-2)
        t0 += n
    batch = lib_batch(w, DEV)
    for _ in range(8):
        sc = torch.empty(batch.score_shape(), device=DEV)
        R.snapkv_score(batch, qw, K, w.W, 1, sc, lse_win=lse)
        assert float(((sc - ref).abs() / ref).max()) < SCORE_RTOL
