"""Small batches split a unit's key chunks over CTAs; the scores are the same
bits as where a chunk is one CTA's: a layer with the workspace it asks for
against the same layer with one that only holds whole chunks, a batch of many
layers (cut less or not at all) against its layers one at a time, and against
the oracle."""

import math

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


# One layer of each is cut on 152 SMs, except where it says so (a chunk of less
# than eight tiles gains nothing).
CASES = {
    "one_cell": _w(40, 2, 4, 128, 512, 32),
    "cell_and_a_tile": _w(40, 2, 4, 128, 513, 32),
    "d64_shorter_than_window": _w(40, 2, 8, 64, 20, 32),
    "two_cells": _w(40, 2, 4, 128, 1024, 32),
    "two_cells_and_a_key": _w(40, 2, 8, 64, 1025, 32),
    "odd_tiles_two_row_tiles": _w(20, 4, 4, 128, 1500, 64),
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
UNCUT = {"one_cell", "cell_and_a_tile", "d64_shorter_than_window"}


def _whole_chunks_bytes(batch):
    """The two-pass workspace of the plan that cuts no chunk."""
    tiles = (batch.n_max + 127) // 128
    nc = max(1, min(8, (tiles + 63) // 64))
    per = max(1, (tiles + nc - 1) // nc)
    chunks = max(1, (tiles + per - 1) // per)
    al = lambda x: (x + 255) // 256 * 256
    units, elems = batch.n_units, math.prod(batch.score_shape())
    return 256 + al(units * chunks * 256 * 8) + al(units * 256 * 4) + al(elems * 4) + al((units + 1) * 4)


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
    # a layer, cut and not
    layer = lib_batch(one, DEV)
    uncut, asked = _whole_chunks_bytes(layer), R.workspace_size(R.OP_SNAPKV, layer, w.W)
    assert (asked == uncut) if name in UNCUT else (asked > uncut)
    small = torch.empty(uncut, dtype=torch.uint8, device=DEV)
    for l in (0, w.L - 1):
        assert torch.equal(parts[l], _score(one, K[l:l + 1], qw[l:l + 1], ws=small))
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


def test_a_workspace_too_small_for_whole_chunks_is_refused():
    w = CASES["two_chunks"].scaled(L=1)
    K, qw = _inputs(w)
    batch = lib_batch(w, DEV)
    sc = torch.empty(batch.score_shape(), device=DEV)
    ws = torch.empty(_whole_chunks_bytes(batch) - 256, dtype=torch.uint8, device=DEV)
    with pytest.raises(R.RolekvError):
        R.snapkv_score(batch, qw, K, w.W, 7, sc, ws=ws)


def test_compression_with_a_workspace_for_whole_chunks():
    """A workspace that only holds whole chunks gives the same kept rows."""
    w = CASES["odd_tiles_two_row_tiles"].scaled(L=1)
    roles = I.workload_roles(w, 4)
    K, V = I.make_kv(w, roles, 4, device=DEV)
    qw = I.make_q_window(w, 4, device=DEV)
    batch = lib_batch(w, DEV)
    params = R.select_params(0.2, I.PAPER_ALPHA, alpha_key=0.02, key_role=I.ROLE_KEY)
    out = []
    for size in (R.workspace_size(R.OP_COMPRESS, batch, w.W), _whole_chunks_bytes(batch)):
        idx = torch.empty(batch.kept_shape(0.2), dtype=torch.int32, device=DEV)
        kv = torch.empty((2,) + R.compact_shape(batch, 0.2), dtype=torch.bfloat16, device=DEV)
        R.rolekv_compress(batch, qw, K, V, w.W, 7, torch.as_tensor(roles, device=DEV), params, idx, kv[0], kv[1],
                          torch.empty(size, dtype=torch.uint8, device=DEV))
        out.append((idx, kv))
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1].view(torch.int16), out[1][1].view(torch.int16))
