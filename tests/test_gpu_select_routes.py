"""The selector's routes (one CTA per unit, a cluster of CTAs per unit,
streaming) give the same kept sets: a batch large enough for one route against
its layers one at a time, which take another, and sampled units against the
oracle."""

import threading

import numpy as np
import pytest
import torch

from oracle import rolekv_oracle as O
from paper_2607_13205_gb300 import inputs as I
from paper_2607_13205_gb300 import rolekv as R
from tests.gpu_helpers import lib_batch, oracle_batch

pytestmark = pytest.mark.gpu

DEV = "cuda"


def _scores(kind, shape, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    x = torch.randn(shape, generator=g, device=DEV)
    if kind == "spread":
        return torch.exp(1.5 * x)
    if kind == "tied":                       # a few hundred values: ties at every threshold
        return torch.exp(torch.round(8 * x) / 16)
    if kind == "constant":                   # every key equal: ties ranked over all slots and ranks
        return torch.full(shape, 0.37, device=DEV)
    if kind == "signs":                      # both signs: the full-pass descent
        return x
    x = torch.exp(x)                         # "nan": a few of them
    x.view(-1)[:: max(1, x.numel() // 7)] = float("nan")
    return x


# (n, layers, policy, pool, budget, floor, scores[, varlen lengths]): the whole
# batch and one layer of it take different routes (4 KV heads a sequence)
CASES = [
    (16385, 10, R.POLICY_ROLE_QUOTA, 7, 0.1, 0, "spread"),
    (16385, 10, R.POLICY_GLOBAL, 1, 0.3, 64, "tied"),
    (20003, 10, R.POLICY_SLACK, 7, 0.3, 32, "spread"),
    (20003, 10, R.POLICY_SLACK, 3, 0.5, 0, "constant"),
    (24001, 10, R.POLICY_ROLE_QUOTA, 5, 0.2, 0, "signs"),
    (24001, 10, R.POLICY_FAIR, 1, 0.5, 0, "constant"),
    (40960, 10, R.POLICY_ROLE_QUOTA, 15, 0.02, 0, "nan"),
    (40961, 20, R.POLICY_ROLE_QUOTA, 7, 0.1, 0, "tied"),
    (40961, 20, R.POLICY_SLACK, 7, 0.3, 0, "tied"),
    (40961, 20, R.POLICY_GLOBAL, 3, 0.1, 16, "constant"),
    (65537, 20, R.POLICY_FAIR, 7, 0.05, 0, "nan"),
    (131137, 10, R.POLICY_GLOBAL, 7, 0.1, 64, "spread"),
    (262144, 10, R.POLICY_ROLE_QUOTA, 7, 0.02, 0, "tied"),
    (132100, 4, R.POLICY_SLACK, 7, 0.2, 0, "tied"),
    (163840, 5, R.POLICY_GLOBAL, 7, 0.1, 32, "spread"),
    (50001, 7, R.POLICY_ROLE_QUOTA, 7, 0.1, 32, "tied", (50001, 3, 0, 17111, 1)),
    (4096, 40, R.POLICY_ROLE_QUOTA, 7, 0.1, 0, "spread"),
    (8192, 160, R.POLICY_SLACK, 7, 0.3, 0, "tied"),
    # positions written by slot where more than 0.39 of a run of words is kept
    (5003, 40, R.POLICY_GLOBAL, 3, 0.6, 5, "spread"),
    (2049, 40, R.POLICY_ROLE_QUOTA, 1, 0.4, 0, "spread"),
    (8191, 2, R.POLICY_SLACK, 7, 0.4, 0, "constant"),
    (45003, 20, R.POLICY_ROLE_QUOTA, 7, 0.5, 0, "spread"),
    (70000, 20, R.POLICY_GLOBAL, 7, 1.0, 0, "tied"),
]


@pytest.mark.parametrize("case", CASES, ids=[f"{c[0]}x{c[1]}-p{c[2]}-{c[6]}" for c in CASES])
def test_routes_agree(case):
    n, L, policy, pool, B, floor, kind = case[:7]
    lens = case[7] if len(case) > 7 else None
    w = I.Workload("routes", "snapkv", L, len(lens) if lens else 1, 8, 4, 64, n, 32, pool, (B,), 4, (3, 5), (1, 3),
                   seqlens=lens)
    one = w.scaled(L=1)
    roles_np = I.workload_roles(w, 3)
    roles = torch.as_tensor(roles_np, device=DEV)
    params = R.select_params(B, I.PAPER_ALPHA, alpha_key=0.02, key_role=I.ROLE_KEY, policy=policy, keep_last=floor)
    whole, layer = lib_batch(w, DEV), lib_batch(one, DEV)
    scores = _scores(kind, whole.score_shape(), 11)

    def run(batch, sc):
        idx = torch.full(batch.kept_shape(B), -7, dtype=torch.int32, device=DEV)
        mask = torch.full(batch.score_shape(), 9, dtype=torch.uint8, device=DEV)
        per = torch.full((batch.n_units, I.N_ROLES), -1, dtype=torch.int32, device=DEV)
        status = torch.zeros(1, dtype=torch.int32, device=DEV)
        R.role_alloc_select(batch, sc, roles, params, idx, pool_k=pool, keep_mask=mask, kept_per_role=per,
                            status=status)
        return idx, mask, per, status

    a = run(whole, scores)
    parts = [run(layer, scores[l:l + 1].contiguous()) for l in range(L)]
    torch.cuda.synchronize()
    for x in range(3):
        assert torch.equal(a[x], torch.cat([p[x] for p in parts], dim=0)), ("idx", "mask", "per_role")[x]
    assert int(a[3]) == (R.STATUS_NONFINITE if kind == "nan" else 0)
    if kind == "nan":
        return                               # (the oracle's NaN rule has its own test)
    # the first layer's units against the oracle
    ob = oracle_batch(one)
    sc = scores[:1].cpu().numpy()
    us = {u: ob.score_view(sc, u).astype(np.float64) for u in range(ob.n_units)}
    us = {u: O.maxpool1d(s, pool) if s.size else s for u, s in us.items()}
    ref = O.select_batch(ob, us, roles_np, I.N_ROLES, I.PAPER_ALPHA, I.ROLE_KEY, 0.02, B, policy, 0, keep_last=floor)
    cu = ob.kept_offsets(B)
    got, per = parts[0][0].cpu().numpy(), parts[0][2].cpu().numpy()
    for u, (idx, counts) in ref.items():
        _, s, h = ob.unit(u)
        row = got[0, h, cu[s]:cu[s + 1]] if ob.varlen else got.reshape(ob.n_units, -1)[u]
        assert np.array_equal(row, idx), f"unit {u}"
        assert list(per[u]) == counts, f"unit {u} per-role counts"


@pytest.mark.parametrize("n,units,role", [(8192, 400, 0), (8192, 8, 3), (40960, 40, 2), (163840, 20, 1), (262144, 48, 3)])
def test_counts_of_one_role_and_everything_kept(n, units, role):
    """The largest share of a role's count that a lane can hold, on each route."""
    batch = R.Batch(units, 1, 1, 1, 64, n)
    roles = torch.full((1, n), role, dtype=torch.uint8, device=DEV)
    params = R.select_params(1.0, I.PAPER_ALPHA, policy=R.POLICY_GLOBAL)
    idx = torch.full(batch.kept_shape(1.0), -7, dtype=torch.int32, device=DEV)
    per = torch.full((units, I.N_ROLES), -1, dtype=torch.int32, device=DEV)
    R.role_alloc_select(batch, torch.rand(units, 1, 1, n, device=DEV), roles, params, idx, kept_per_role=per)
    assert torch.equal(idx, torch.arange(n, dtype=torch.int32, device=DEV).expand_as(idx))
    assert per.tolist() == [[n if r == role else 0 for r in range(I.N_ROLES)]] * units


@pytest.mark.parametrize("sizes", [((40960, 76), (20000, 76)), ((131072, 8), (70000, 8)), ((40960, 8), (17000, 8))],
                         ids=["one", "cluster", "cluster_512"])
def test_two_threads_with_rows_of_different_lengths(sizes):
    """Calls of the same kernel with more and less shared memory from two
    threads at once: neither is refused for the other's limit."""
    errors = []

    def work(n, units):
        try:
            batch = R.Batch(units, 1, 1, 1, 64, n)
            g = torch.Generator(device=DEV).manual_seed(n)
            scores = torch.rand(batch.score_shape(), generator=g, device=DEV)
            roles = torch.zeros((1, n), dtype=torch.uint8, device=DEV)
            params = R.select_params(0.1, I.PAPER_ALPHA, policy=R.POLICY_GLOBAL)
            s = torch.cuda.Stream()
            s.wait_stream(torch.cuda.current_stream())
            idx = [torch.empty(batch.kept_shape(0.1), dtype=torch.int32, device=DEV) for _ in range(2)]
            for i in range(1500):
                R.role_alloc_select(batch, scores, roles, params, idx[i > 0], stream=s)
            s.synchronize()
            assert torch.equal(idx[0], idx[1])
        except Exception as e:                       # noqa: BLE001  (reported by the main thread)
            errors.append(repr(e))

    threads = [threading.Thread(target=work, args=x) for x in sizes]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
