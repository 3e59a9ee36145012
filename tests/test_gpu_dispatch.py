"""Every branch of the size-dependent dispatch rules, at the sizes where each can go wrong, against the CPU oracle."""
import numpy as np
import pytest
import torch

import oracle
import synth_inputs as si
from harness import A, Case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [1, 2, 3, 4, 5, 6, 7, 8, 9, 13, 16])
def test_calibration_sums_by_top_k(K):
    """Pair sums: a kernel per Top-K up to 8, tiles of four slots above (9: a ragged last tile). d = 132 leaves a tail
    after whole 128-column steps; m is not a multiple of the tokens per block. fp32 outputs, double sums: the oracle's
    tables to fp32 rounding of the outputs (2e-5, as in the other fp32 calibration tests)."""
    N = 16
    cfg = si.LayerConfig("calk", N, 0, 132, 64, K, "f32", 16, (1,), 4, (2,))
    case = Case(cfg, std=0.05, correlated=0.8)
    m = 61
    xc, lc = si.hidden_states(cfg, m, "x_cal"), si.router_logits(cfg, m, "logits_cal")
    ref = oracle.calibrate(A(xc), lc.numpy(), A(case.wg), A(case.wu), A(case.wd), N, K, mode=0)
    dev, ex = case.dev, case.ex
    S, L = torch.empty((N, N), device=dev), torch.empty((N, N), device=dev)
    h, lnh, n_obs = torch.empty(N, device=dev), torch.empty(N, device=dev), torch.empty((N, N), dtype=torch.int32, device=dev)
    ws = ex.alloc_workspace(case.layer, m, K)
    ws.fill_(0xFF)
    rc = ex.exfold_calibrate(case.layer, xc.to(dev), lc.to(dev), case.d_wg, case.d_wu, case.d_wd,
                             ex.make_tables(S, L, h, lnh, n_obs), ws)
    assert rc == (1 if ref["unobserved"] else 0)
    assert np.array_equal(n_obs.cpu().numpy(), ref["n_obs"])
    np.testing.assert_allclose(S.cpu().numpy(), ref["S"], rtol=2e-5, atol=2e-6)
    np.testing.assert_allclose(L.cpu().numpy(), ref["L"], rtol=1e-4, atol=2e-5)
    np.testing.assert_allclose(h.cpu().numpy(), ref["h"], rtol=1e-5)
    np.testing.assert_allclose(lnh.cpu().numpy(), ref["lnh"], rtol=1e-5, atol=1e-6)
