"""NaN and infinite values that a call meets: what they may touch and what they may not."""
import numpy as np
import pytest
import torch

import synth_inputs as si
from harness import Case, check_decode_meta, check_output

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
