"""The standalone max-pool (16-byte groups) at row starts and ends of every
alignment and every width, 1 (a plain copy) included."""

import pytest
import torch

from paper_2607_13205_gb300 import inputs as I
from paper_2607_13205_gb300 import rolekv as R
from tests.gpu_helpers import lib_batch

pytestmark = pytest.mark.gpu

DEV = "cuda"


@pytest.mark.parametrize("pool", [1, 3, 5, 7, 9, 11, 13, 15])
@pytest.mark.parametrize("lens", [(1, 2, 3, 5), (1023, 1, 1025, 4), None])
def test_pool_matches_window_maximum(pool, lens):
    n = max(lens) if lens else 1021
    w = I.Workload("pool", "snapkv", 2, len(lens) if lens else 3, 4, 2, 64, n, 8, pool, (0.1,), 4, (3, 5), (1, 3),
                   seqlens=lens)
    roles = I.workload_roles(w, 1)
    K, _ = I.make_kv(w, roles, 1, device=DEV, with_v=False)
    qw = I.make_q_window(w, 1, device=DEV)
    batch = lib_batch(w, DEV)
    # (scores one element into their buffer: the output rows' alignment differs from the inputs')
    numel = 1
    for x in batch.score_shape():
        numel *= x
    pre = torch.empty(batch.score_shape(), device=DEV)
    out = torch.full((numel + 1,), -7.0, device=DEV)[1:].view(batch.score_shape())
    R.snapkv_score(batch, qw, K, w.W, pool, out, scores_prepool=pre)
    torch.cuda.synchronize()
    rows, got, t0 = [], [], 0
    for s, m in enumerate(w.lengths()):
        rows.append(pre[:, :, t0:t0 + m] if w.varlen else pre[:, s])
        got.append(out[:, :, t0:t0 + m] if w.varlen else out[:, s])
        t0 += m
    for x, y in zip(rows, got):
        ref = torch.nn.functional.max_pool1d(x, pool, stride=1, padding=pool // 2)
        assert torch.equal(y, ref)
