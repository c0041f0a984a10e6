"""Small batches split a unit's key chunks over CTAs; the scores are the same
bits as where a chunk is one CTA's: a batch too large for the split against
its layers one at a time, and against the oracle."""

import pytest
import torch

from oracle import rolekv_oracle as O
from paper_2607_13205_gb300 import inputs as I
from paper_2607_13205_gb300 import rolekv as R
from tests.gpu_helpers import assert_scores_close, lib_batch, oracle_batch

pytestmark = pytest.mark.gpu

DEV = "cuda"


def _w(L, Hkv, G, d, n, W, lens=None):
    return I.Workload("split", "snapkv", L, len(lens) if lens else 1, Hkv * G, Hkv, d, n, W, 7, (0.1,), 4, (3, 5),
                      (1, 3), seqlens=lens)


# the whole batch has more than 76 chunks (no split), a layer at most 20
CASES = {
    "one_cell": _w(40, 2, 4, 128, 512, 32),
    "cell_and_a_tile": _w(40, 2, 4, 128, 513, 32),
    "odd_tiles_two_row_tiles": _w(20, 4, 4, 128, 1500, 64),
    "d64_shorter_than_window": _w(40, 2, 8, 64, 20, 32),
    "g7_padded_rows": _w(20, 4, 7, 128, 2177, 32),
    "two_chunks": _w(10, 4, 4, 128, 8500, 32),
    "eight_chunks": _w(4, 4, 2, 64, 66000, 64),
    "varlen": _w(7, 4, 4, 128, 3000, 32, (3000, 0, 1, 700)),
    # (several rounds of items a CTA)
    "rounds_g1_8_rows": _w(40, 2, 1, 128, 2500, 8),
    "rounds_d64": _w(100, 4, 4, 64, 5000, 32),
    "rounds_32_cells": _w(12, 8, 2, 128, 16384, 64),
    "rounds_empty_last_part": _w(80, 4, 3, 128, 2561, 40),
    "rounds_varlen": _w(40, 2, 4, 128, 4000, 32, (4000, 1, 0, 1030, 2300)),
    "varlen_chunks_g7": _w(7, 4, 7, 128, 9000, 32, (9000, 129, 5000)),
}


def _inputs(w):
    roles = I.workload_roles(w, 4)
    K, _ = I.make_kv(w, roles, 4, device=DEV, with_v=False)
    return K, I.make_q_window(w, 4, device=DEV)


def _score(w, K, qw, **kw):
    b = lib_batch(w, DEV)
    sc = torch.full(b.score_shape(), -1.0, dtype=torch.float32, device=DEV)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    R.snapkv_score(b, qw, K, w.W, 1, sc, status=status, **kw)
    torch.cuda.synchronize()
    assert int(status) == 0
    return sc


@pytest.mark.parametrize("name", CASES)
def test_split_scores_match_whole_chunks(name):
    w = CASES[name]
    K, qw = _inputs(w)
    whole = _score(w, K, qw)
    one = w.scaled(L=1)
    parts = [_score(one, K[l:l + 1], qw[l:l + 1]) for l in range(w.L)]
    assert torch.equal(whole, torch.cat(parts, dim=0))
    # with supplied normalisers: pass 2 alone, split or not
    lse = 0.5 + torch.rand(w.L, w.b, w.Hq, w.W, device=DEV)
    whole = _score(w, K, qw, lse_win=lse)
    parts1 = [_score(one, K[l:l + 1], qw[l:l + 1], lse_win=lse[l:l + 1].contiguous()) for l in range(w.L)]
    assert torch.equal(whole, torch.cat(parts1, dim=0))
    ob = oracle_batch(one)
    ref = O.snapkv_batch(ob, I.bf16_bits(qw[:1]), I.bf16_bits(K[:1]), w.W, 1)
    got = parts[0].cpu().numpy()
    for u, (pre, _) in ref.items():
        assert_scores_close(ob.score_view(got, u), pre, f"{name} unit {u}")


def test_workspace_of_the_unsplit_plan_is_accepted():
    """A workspace too small for the split's partials is used without it."""
    w = CASES["two_chunks"].scaled(L=1)
    K, qw = _inputs(w)
    batch = lib_batch(w, DEV)
    full = R.workspace_size(R.OP_SNAPKV, batch, w.W)
    al = lambda x: (x + 255) // 256 * 256
    units, chunks = batch.n_units, 2
    need = 256 + al(units * chunks * 256 * 8) + al(units * 256 * 4) + al(units * w.n * 4) + al((units + 1) * 4)
    assert need < full
    a = _score(w, K, qw)
    b = _score(w, K, qw, ws=torch.empty(need, dtype=torch.uint8, device=DEV))
    assert torch.equal(a, b)
    sc = torch.empty(batch.score_shape(), device=DEV)
    with pytest.raises(R.RolekvError):
        R.snapkv_score(batch, qw, K, w.W, 7, sc, ws=torch.empty(need - 256, dtype=torch.uint8, device=DEV))
