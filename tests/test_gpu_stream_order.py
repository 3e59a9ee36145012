"""Inputs that the caller writes on the stream right before a call."""
import numpy as np
import pytest
import torch

import oracle
import synth_inputs as si
from harness import Case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,router", [(1, False), (8, False), (8, True), (9, False), (64, True), (200, False)])
def test_tables_written_right_before_the_call(B, router):
    """A kernel that changes the norm table, then the decode call, 24 times without a synchronisation: every call's pool is
    that of its own norms (the calls' first kernels may start before the caller's kernel has ended)."""
    N, K, M, d = 128, 4, 6, 256
    case = Case(si.LayerConfig("order", N, 0, d, 64, K, "bf16", 8, (1,), B, (M,)))
    ex, dev = case.ex, case.dev
    S, L, h, _ = case.tables_host
    wr = si.router_weights(case.cfg).to(dev)
    lg = torch.empty((B, N), device=dev)
    norms = [h[torch.from_numpy(np.random.default_rng(i).permutation(N))].contiguous() for i in range(2)]
    d_norms = [t.to(dev) for t in norms]
    y = torch.empty((B, d), dtype=torch.bfloat16, device=dev)
    pools = torch.full((24, M), -7, dtype=torch.int32, device=dev)
    ws = case.workspace(B, K)
    busy = torch.empty(1 << 22, device=dev)
    torch.cuda.synchronize()
    for i in range(24):
        busy.mul_(1.0)  # keeps the stream ahead of the host, so that the kernels below queue up
        case.d_tabs[2].copy_(d_norms[i % 2])
        if router:
            ex.exfold_moe_decode_layer(case.layer, case.d_xd, wr, case.d_wg, case.d_wu, case.d_wd, case.tables, M, y, ws, lg,
                                       meta=dict(pool_ids=pools[i]))
        else:
            ex.exfold_moe_decode(case.layer, case.d_xd, case.d_lgd, case.d_wg, case.d_wu, case.d_wd, case.tables, M, y, ws,
                                 meta=dict(pool_ids=pools[i]))
    assert ex.exfold_device_status(ws) == 0
    scores = (lg if router else case.d_lgd).cpu().numpy()
    want = [oracle.decode_fold(scores, K, M, S.numpy(), L.numpy(), t.numpy())["pool_ids"][:M] for t in norms]
    assert not np.array_equal(want[0], want[1])
    got = pools.cpu().numpy()
    for i in range(24):
        assert np.array_equal(got[i], want[i % 2]), i


@pytest.mark.parametrize("op,dtype,T", [("prefill", "bf16", 1), ("prefill", "bf16", 8), ("prefill", "bf16", 40), ("prefill", "f32", 1),
                                        ("prefill", "f32", 64), ("prefill", "f32", 300), ("decode", "f32", 1), ("decode", "f32", 16),
                                        ("decode", "f32", 200), ("decode", "bf16", 5)])
def test_inputs_written_right_before_the_call(op, dtype, T):
    """Kernels that change the tables, the scores and x, then the call, 24 times without a synchronisation: the kernel that routes
    first (the FFN kernel itself for few tokens) reads what was written, and each call has the bits of one alone."""
    N, K, Kp, M, d = 24, 4, 2, 5, 256
    case = Case(si.LayerConfig("order2", N, 0, d, 64, K, dtype, T, (Kp,), T, (M,)))
    ex, dev = case.ex, case.dev
    sets = [[t.clone() for t in (*case.d_tabs, case.d_x, case.d_lg)]]
    perm = torch.from_numpy(np.random.default_rng(3).permutation(N)).to(dev)
    S, L, h, lnh, x, lg = sets[0]
    sets.append([S[perm][:, perm].contiguous(), L[perm][:, perm].contiguous(), h[perm].contiguous(), lnh[perm].contiguous(), -x, lg[:, perm].contiguous()])
    live = [t.clone() for t in sets[0]]
    tables = ex.make_tables(*live[:4])
    ws = case.workspace(T, K)
    ys = torch.full((24, T, d), float("nan"), dtype=case.d_wg.dtype, device=dev)

    def call(i):
        for t, v in zip(live, sets[i % 2]):
            t.copy_(v)
        if op == "decode":
            ex.exfold_moe_decode(case.layer, live[4], live[5], case.d_wg, case.d_wu, case.d_wd, tables, M, ys[i], ws)
        else:
            ex.exfold_moe_prefill(case.layer, live[4], live[5], case.d_wg, case.d_wu, case.d_wd, tables, Kp, ys[i], ws)

    want = []
    for i in range(2):
        call(i)
        torch.cuda.synchronize()
        want.append(ys[i].clone())
    assert not torch.equal(want[0], want[1])
    ys.fill_(float("nan"))
    busy = torch.empty(1 << 22, device=dev)
    torch.cuda.synchronize()
    for i in range(24):
        busy.mul_(1.0)  # keeps the stream ahead of the host
        call(i)
    assert ex.exfold_device_status(ws) == 0
    for i in range(24):
        assert torch.equal(ys[i], want[i % 2]), i
