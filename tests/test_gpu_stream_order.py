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
