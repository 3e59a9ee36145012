"""NaN and infinite values that a call meets: what they may touch and what they may not."""
import numpy as np
import pytest
import torch

import oracle
import synth_inputs as si
from harness import A, Case, check_decode_meta, check_output

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B", [3, 8, 20, 140])
@pytest.mark.parametrize("N,M", [(16, 1), (40, 3), (40, 12), (200, 70)])
def test_decode_targets_of_nan_losses(B, N, M):
    """Eq. 12 over losses of which a third are NaN or infinite, some sources' all: a NaN is never smaller, and one at the
    best-ranked pool expert, where the search starts, stays. Targets and scalars as the oracle's, bit for bit."""
    case = Case(si.LayerConfig("nanloss", N, 0, 128, 64, 4, "bf16", 8, (1,), B, (M,)))
    S, L, h, lnh = case.tables_host
    rng = np.random.default_rng(B + N + M)
    L = L.clone()
    L[torch.from_numpy(rng.uniform(size=(N, N)) < 0.3)] = float("nan")
    L[torch.from_numpy(rng.uniform(size=(N, N)) < 0.05)] = float("inf")
    L[::5] = float("nan")
    L[1::5] = float("inf")
    case.set_tables((S, L, h, lnh))
    got, ref = case.run_decode(M), case.oracle_decode(M)
    check_decode_meta(got, ref, M)
    check_output(got["y"], ref["y"], "bf16")
    plain = case.run_decode(M, with_meta=False)  # without metadata only the batch's experts get targets
    assert np.array_equal(got["y"], plain["y"])


@pytest.mark.parametrize("T", [1, 2, 5, 8, 9, 40, 130])
@pytest.mark.parametrize("dtype,ns", [("bf16", 0), ("bf16", 1), ("f32", 0)])
@pytest.mark.parametrize("bad", [float("inf"), float("nan")])
def test_a_broken_expert_touches_its_own_tokens_only(T, dtype, ns, bad):
    """One non-finite weight in one expert: the outputs of tokens that are not routed to it keep their bits, those of its
    own tokens are not finite. Prefill, decode with the dynamic and the static pool; gate, up and down weights in turn."""
    N, K, d, I = 12, 2, 192, 320
    case = Case(si.LayerConfig("broken", N, ns, d, I, K, dtype, T, (K,), T, (N,)))
    ex, dev = case.ex, case.dev
    for lg in (case.lg, case.lgd):  # expert 3 serves every third token, the first among them
        lg[:, 3] = torch.where(torch.arange(T) % 3 == 0, 9.0, -9.0)
    case.d_lg, case.d_lgd = case.lg.to(dev), case.lgd.to(dev)
    case.d_x, case.d_xd = case.d_x.abs() + 0.5, case.d_xd.abs() + 0.5  # no zero meets the bad weight
    pool = [torch.empty(N, dtype=torch.int32, device=dev), torch.empty(N, dtype=torch.int32, device=dev), torch.empty(N, device=dev)]
    sp = ex.exfold_static_pool_build(case.layer, case.tables, N, *pool)

    def static():
        y = torch.full((T, d), float("nan"), dtype=case.d_wg.dtype, device=dev)
        ws = case.workspace(T, K)
        ex.exfold_moe_decode_static(case.layer, case.d_xd, case.d_lgd, case.d_wg, case.d_wu, case.d_wd, sp, y, ws)
        return y.float().cpu().numpy()

    runs = [lambda: case.run_prefill(K, with_meta=False)["y"], lambda: case.run_decode(N, with_meta=False)["y"], static]
    clean = [run() for run in runs]
    mine = np.arange(T) % 3 == 0
    for w in (case.d_wg, case.d_wu, case.d_wd):
        keep = w[3, 5, 7].clone()
        w[3, 5, 7] = bad
        for run, want in zip(runs, clean):
            got = run()
            assert np.array_equal(got[~mine], want[~mine])
            if bad != bad or w is not case.d_wg:  # (an infinite gate may be silu(-inf) = 0 or x - inf)
                assert not np.isfinite(got[mine]).all(axis=1).any()
        w[3, 5, 7] = keep


def check_routing_is_whole(got, T, K, Kp, N):
    """Whatever the scores: Kp distinct experts per token, the omitted ones beside them, every route sorted once."""
    routes = np.concatenate([got["ids"], got["omit_src"]], axis=1)
    assert routes.min() >= 0 and routes.max() < N
    assert all(len(set(r)) == K for r in routes.tolist())
    assert np.array_equal(np.diff(got["offsets"]), np.bincount(got["ids"].ravel(), minlength=N))
    assert got["offsets"][0] == 0 and np.array_equal(np.sort(got["perm"]), np.arange(T * Kp))


@pytest.mark.parametrize("dtype,ns,N", [("bf16", 0, 12), ("bf16", 1, 40), ("f32", 0, 12), ("f32", 1, 140)])
@pytest.mark.parametrize("T,K,Kp", [(1, 4, 2), (3, 4, 4), (8, 6, 3), (9, 4, 3), (64, 5, 2), (128, 4, 4), (300, 4, 2), (2300, 3, 2)])
def test_prefill_tokens_of_non_finite_scores(T, K, Kp, dtype, ns, N):
    """Scores of every third token NaN (of either sign), infinite or one of them, and a NaN norm: each token has its K' distinct
    retained routes and the others keep their bits, with the metadata and without."""
    case = Case(si.LayerConfig("nanscore", N, ns, 128, 192, K, dtype, T, (Kp,), 4, (2,)))
    lg = case.lg.clone()
    want = case.run_prefill(Kp)
    bad = np.arange(T) % 3 == 0
    kinds = [torch.full((N,), float("nan")), torch.full((N,), -float("nan")), torch.full((N,), float("inf")),
             torch.full((N,), float("-inf")), torch.where(torch.arange(N) % 2 == 0, float("nan"), 1.0),
             torch.where(torch.arange(N) == 5, float("inf"), 0.0), torch.where(torch.arange(N) % 3 == 0, -float("nan"), float("nan"))]
    for j, i in enumerate(np.flatnonzero(bad)):
        case.lg[i] = kinds[(j + T) % len(kinds)]
    case.d_lg = case.lg.to(case.dev)
    got = case.run_prefill(Kp)
    check_routing_is_whole(got, T, K, Kp, N)
    assert np.array_equal(got["y"][~bad], want["y"][~bad])
    assert np.array_equal(got["y"], case.run_prefill(Kp, with_meta=False)["y"], equal_nan=True)
    # a norm: its expert's tokens are folded in some order, the others' bits stay
    case.d_lg = lg.to(case.dev)
    S, L, h, lnh = (t.clone() for t in case.tables_host)
    h[2] = lnh[2] = float("nan")
    case.set_tables((S, L, h, lnh))
    got = case.run_prefill(Kp)
    check_routing_is_whole(got, T, K, Kp, N)
    clean = (lg.topk(K, dim=1).indices != 2).all(dim=1).numpy()
    assert np.array_equal(got["y"][clean], want["y"][clean])


def bad_scores(lgd):
    """Every fourth token's scores NaN or infinite, in part or in whole; which tokens."""
    B, N = lgd.shape
    kinds = [torch.full((N,), float("nan")), torch.full((N,), float("inf")), torch.full((N,), float("-inf")),
             torch.where(torch.arange(N) % 2 == 0, -float("nan"), 1.0)]
    bad = np.arange(B) % 4 == 2
    for j, i in enumerate(np.flatnonzero(bad)):
        lgd[i] = kinds[j % len(kinds)]
    return bad


@pytest.mark.parametrize("dtype,ns,N", [("bf16", 0, 24), ("bf16", 1, 200), ("f32", 0, 24), ("f32", 1, 120), ("f32", 0, 140)])
@pytest.mark.parametrize("B", [1, 3, 8, 20, 60, 129, 200])
@pytest.mark.parametrize("M", [1, 5, 20])
def test_decode_pool_of_non_finite_norms(B, M, dtype, ns, N):
    """A third of the norms NaN or infinite and some tokens' scores too: a pool of distinct experts of the batch, every route on one
    of them, and the tokens of finite scores are the sums over the routes that the metadata names."""
    K = 4
    case = Case(si.LayerConfig("nannorm", N, ns, 128, 192, K, dtype, 8, (1,), B, (M,)))
    S, L, h, lnh = (t.clone() for t in case.tables_host)
    h[::3], h[1::7], h[2::11] = float("nan"), float("inf"), -float("nan")
    case.set_tables((S, L, h, lnh))
    bad = bad_scores(case.lgd)
    case.d_lgd = case.lgd.to(case.dev)
    got = case.run_decode(M)
    P, pool = int(got["pool_size"][0]), got["pool_ids"]
    assert 1 <= P <= M and len(set(pool[:P].tolist())) == P and pool[:P].min() >= 0 and pool[:P].max() < N and (pool[P:] == -1).all()
    mask = got["pool_mask"].view(np.uint32)
    assert sorted(pool[:P].tolist()) == [e for e in range(N) if mask[e >> 5] >> (e & 31) & 1]
    assert np.isin(got["ids"], pool[:P]).all() and np.isin(got["target"], pool[:P]).all()
    assert np.array_equal(got["y"], case.run_decode(M, with_meta=False)["y"], equal_nan=True)
    yr = oracle.moe_apply(A(case.xd), A(case.wg), A(case.wu), A(case.wd), got["ids"], np.where(bad[:, None], 0, got["w"]).astype(np.float32), N, ns)
    check_output(got["y"][~bad], yr[~bad], dtype)


@pytest.mark.parametrize("dtype,N,B", [("bf16", 24, 5), ("bf16", 200, 40), ("bf16", 24, 200), ("f32", 24, 40), ("f32", 140, 40)])
@pytest.mark.parametrize("M", [1, 5, 20])
def test_static_pool_of_non_finite_norms(M, dtype, N, B):
    """The static pool built from norms of which a third are NaN or infinite: M distinct experts, every target among them; a step on
    it is the sum over the remapped routes."""
    K, d = 4, 128
    case = Case(si.LayerConfig("nanstat", N, 0, d, 192, K, dtype, 8, (1,), B, (M,)))
    ex, dev = case.ex, case.dev
    S, L, h, lnh = (t.clone() for t in case.tables_host)
    h[::3], h[1::7], h[2::11] = float("nan"), float("inf"), -float("nan")
    case.set_tables((S, L, h, lnh))
    pool_t = [torch.full((M,), -7, dtype=torch.int32, device=dev), torch.full((N,), -7, dtype=torch.int32, device=dev), torch.empty(N, device=dev)]
    pool = ex.exfold_static_pool_build(case.layer, case.tables, M, *pool_t)
    ids, target, scale = (t.cpu().numpy() for t in pool_t)
    assert len(set(ids.tolist())) == M and ids.min() >= 0 and ids.max() < N
    assert np.isin(target, ids).all() and np.array_equal(target[ids], ids)
    out, w = torch.empty((B, K), dtype=torch.int32, device=dev), torch.empty((B, K), device=dev)
    y, ws = torch.full((B, d), float("nan"), dtype=case.d_wg.dtype, device=dev), case.workspace(B, K)
    ex.exfold_moe_decode_static(case.layer, case.d_xd, case.d_lgd, case.d_wg, case.d_wu, case.d_wd, pool, y, ws, meta=dict(ids=out, w=w))
    assert ex.exfold_device_status(ws) == 0
    assert np.array_equal(out.cpu().numpy(), target[case.lgd.topk(K, dim=1).indices.numpy()])
    yr = oracle.moe_apply(A(case.xd), A(case.wg), A(case.wu), A(case.wd), out.cpu().numpy(), w.cpu().numpy(), N, 0)
    check_output(y.float().cpu().numpy(), yr, dtype)
