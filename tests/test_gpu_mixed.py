"""Whole row tiles and ragged remainders in one pass (gemm_mixed.cu), at the group sizes where it can go wrong: against the
one-CTA kernel bit for bit (the same products accumulated in the same order) and against the CPU oracle. MIXED forces the pass, so
that the sizes here do not hang on the library's choice, which has a test of its own."""
import numpy as np
import pytest
import torch

import oracle
import synth_inputs as si
from harness import A, Case, check_output, check_prefill_meta

pytestmark = pytest.mark.gpu
ONE_CTA, PAIRS, MIXED = 1, 2, 3  # gemm_path

EDGES = [0, 1, 2, 31, 32, 33, 63, 64, 65, 96, 97, 127, 128, 129, 160, 161, 192, 193, 223, 224, 225, 255, 256, 257, 288, 289, 383, 384,
         480, 481, 511, 512, 513, 767, 768, 769]


def mixed_ran(N, ns, d, I, K, Kp, T, gemm_path=0):
    """Whether a call ran the pass: it draws its items from the two work counters in the status record (words 4 and 5), which the
    other kernels leave as they were. (Zero weights: only the routing has to be real.)"""
    from paper_2608_24938_b200 import binding as ex
    dev = torch.device("cuda:0")
    bf16 = dict(dtype=torch.bfloat16, device=dev)
    layer = ex.make_layer(N, ns, d, I, K, "bf16")
    tabs = [torch.zeros(s, device=dev) for s in ((N, N), (N, N), (N,), (N,))]
    wg, wu, wd = torch.zeros((N + ns, I, d), **bf16), torch.zeros((N + ns, I, d), **bf16), torch.zeros((N + ns, d, I), **bf16)
    ws = ex.alloc_workspace(layer, T, Kp).fill_(0xFF)
    ex.exfold_moe_prefill_ex(layer, torch.zeros((T, d), **bf16), torch.randn((T, N), device=dev), wg, wu, wd, ex.make_tables(*tabs), Kp,
                             torch.empty((T, d), **bf16), ws, gemm_path=gemm_path)
    torch.cuda.synchronize()
    return ws[16:24].view(torch.int32).tolist() != [-1, -1]


@pytest.mark.parametrize("shape", [(64, 0, 192, 64, 2, 1, 200), (8, 1, 1024, 7168, 3, 2, 2100)])
def test_gemm_path_forces_the_pass(shape):
    """The counters move with MIXED, whatever the size, and with no other forced path."""
    assert mixed_ran(*shape, MIXED) and not mixed_ran(*shape, ONE_CTA) and not mixed_ran(*shape, PAIRS)


@pytest.mark.parametrize("shape,want", [
    # N, shared, d, I, K, K', T
    ((64, 0, 2048, 896, 2, 1, 1536), True),   # 24 rows per expert
    ((64, 0, 2048, 896, 2, 1, 1535), False),
    ((64, 0, 2048, 768, 2, 1, 1536), False),  # fewer than three items per SM
    ((64, 0, 3072, 896, 2, 1, 20), True),     # 48 k-blocks: any number of rows
    ((150, 0, 1024, 320, 2, 1, 21600), True), # 9 k-blocks: 144 rows
    ((150, 0, 1024, 320, 2, 1, 21599), False),
    ((112, 0, 512, 512, 2, 1, 35840), True),  # 8: 320 rows
    ((112, 0, 512, 512, 2, 1, 35839), False),
    ((64, 0, 192, 896, 2, 1, 32000), False),  # fewer: 500 rows are not enough
    ((8, 1, 1024, 7168, 3, 2, 3071), True),   # fewer than eight row tiles per expert
    ((8, 1, 1024, 7168, 3, 2, 3072), False),
])
def test_the_librarys_choice(shape, want):
    """use_mixed on both sides of each of its lines (148 SMs)."""
    assert mixed_ran(*shape) == want


@pytest.mark.parametrize("n_groups", [5, 64])
@pytest.mark.parametrize("d,I", [(64, 64), (64, 896), (320, 832), (1088, 64 * 13), (192, 128)])
def test_group_sizes_at_the_edges_of_tiles(d, I, n_groups):
    """One route per token, dealt so that the experts own exactly the sizes above: one k-block, K and N tails, one column tile, column
    tiles of which the second CTA has none, groups without rows, fewer items than CTA pairs."""
    sizes = EDGES[-5:] if n_groups == 5 else (EDGES * 2)[:64]
    T, N = sum(sizes), len(sizes)
    case = Case(si.LayerConfig("edges", N, 0, d, I, 2, "bf16", T, (1,), 4, (2,)))
    owner = np.repeat(np.arange(N), sizes)[np.random.default_rng(3).permutation(T)]
    lg = torch.full((T, N), -4.0)
    lg[torch.arange(T), torch.from_numpy(owner)] = 4.0
    lg[torch.arange(T), torch.from_numpy((owner + 1) % N)] = -3.0
    case.lg, case.d_lg = lg, lg.to(case.dev)
    case.set_tables((case.tables_host[0], case.tables_host[1], torch.ones(N), torch.zeros(N)))
    got, one = case.run_prefill(1, gemm_path=MIXED), case.run_prefill(1, with_meta=False, gemm_path=ONE_CTA)["y"]
    assert np.array_equal(np.diff(got["offsets"]), sizes)
    assert np.array_equal(got["y"], one)
    idx = np.random.default_rng(4).choice(T, 300, replace=False)
    check_output(got["y"][idx], case.oracle_prefill(1, tok_idx=idx)["y"], "bf16")


@pytest.mark.parametrize("T", [2000, 2048, 2049, 2170])
def test_shared_expert_beside_the_scatter_kernel(T):
    """A shared expert whose gate/up pairs run on the second stream: the pass takes what is left of its group (an odd last row
    tile, or nothing), and all of it in the down projection."""
    case = Case(si.LayerConfig("shared", 8, 1, 1024, 7168, 3, "bf16", T, (2,), 4, (2,)))
    got, one = case.run_prefill(2, gemm_path=MIXED), case.run_prefill(2, with_meta=False, gemm_path=ONE_CTA)["y"]
    assert np.array_equal(got["y"], one)
    idx = np.random.default_rng(5).choice(T, 24, replace=False)
    check_output(got["y"][idx], case.oracle_prefill(2, tok_idx=idx)["y"], "bf16")


@pytest.mark.parametrize("Kp,ns,T,d", [(2, 0, 4000, 192), (3, 1, 2500, 128), (3, 0, 40, 3136), (4, 1, 9, 64)])
def test_rows_of_several_routes(Kp, ns, T, d):
    """Several routes per token through the per-route buffer; few rows of a wide layer."""
    case = Case(si.LayerConfig("routes", 64, ns, d, 896, 4, "bf16", T, (Kp,), 4, (2,), logits="zipf"))
    got, ref = case.run_prefill(Kp, gemm_path=MIXED), case.oracle_prefill(Kp, tok_idx=np.arange(min(T, 200)))
    check_prefill_meta(got, ref)
    check_output(got["y"][:200], ref["y"], "bf16")
    assert np.array_equal(got["y"], case.run_prefill(Kp, with_meta=False, gemm_path=ONE_CTA)["y"])


@pytest.mark.parametrize("mode,m", [(0, 1660), (1, 820), (1, 993)])
def test_calibration(mode, m):
    """fp32 rows of whole and ragged items (820 = 3 x 256 + 52; 993: a rest of 225 rows, a whole item) in a calibration that takes the
    pass: the oracle's tables, tolerances as in test_calibrate_bf16_on_tensor_cores."""
    cfg = si.LayerConfig("calib", 8, 0, 384, 2432, 4, "bf16", 64, (2,), 4, (2,))
    case = Case(cfg, correlated=0.8)
    ex, dev, N = case.ex, case.dev, cfg.n_experts
    xc, lc = si.hidden_states(cfg, m, "x_cal"), si.router_logits(cfg, m, "logits_cal")
    ref = oracle.calibrate(A(xc), lc.numpy(), A(case.wg), A(case.wu), A(case.wd), N, cfg.top_k, mode=mode)
    S = torch.full((N, N), float("nan"), device=dev)
    L, h, lnh = torch.full_like(S, float("nan")), torch.full((N,), float("nan"), device=dev), torch.empty(N, device=dev)
    n_obs = torch.full((N, N), -1, dtype=torch.int32, device=dev)
    ws = ex.alloc_workspace(case.layer, m, N if mode else cfg.top_k)
    ws.fill_(0xFF)
    ex.exfold_calibrate(case.layer, xc.to(dev), lc.to(dev), case.d_wg, case.d_wu, case.d_wd, ex.make_tables(S, L, h, lnh, n_obs), ws, mode=mode)
    assert min(ws[16:24].view(torch.int32).tolist()) > 0  # the pass's work counters
    assert ex.exfold_device_status(ws) == 0
    assert np.array_equal(n_obs.cpu().numpy(), ref["n_obs"])
    np.testing.assert_allclose(S.cpu().numpy(), ref["S"], rtol=5e-3, atol=5e-3)
    seen = (ref["n_obs"] > 0) | np.eye(N, dtype=bool)
    np.testing.assert_allclose(L.cpu().numpy()[seen], ref["L"][seen], rtol=5e-3, atol=5e-3)
    np.testing.assert_allclose(h.cpu().numpy(), ref["h"], rtol=3e-3)


@pytest.mark.parametrize("ns", [0, 1])
def test_two_streams_and_a_replayed_graph(ns):
    """The work counters lie in the workspace and start at zero in every call: calls of one thread on two streams, and a captured
    call replayed, give the bits of the one-CTA kernel."""
    T, Kp = 2049, 2
    case = Case(si.LayerConfig("graph", 8, ns, 1024, 7168, 3, "bf16", T, (Kp,), 4, (2,)))
    ex, dev = case.ex, case.dev
    want = case.run_prefill(Kp, with_meta=False, gemm_path=ONE_CTA)["y"]
    need = ex.exfold_workspace_bytes(case.layer, T, Kp)
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    wss = [torch.full((need,), 0xFF, dtype=torch.uint8, device=dev) for _ in streams]
    ys = [torch.full((T, 1024), float("nan"), dtype=torch.bfloat16, device=dev) for _ in streams]

    def call(i):
        ex.exfold_moe_prefill_ex(case.layer, case.d_x, case.d_lg, case.d_wg, case.d_wu, case.d_wd, case.tables, Kp, ys[i], wss[i],
                                 gemm_path=MIXED, stream=streams[i])

    torch.cuda.synchronize()
    for _ in range(2):
        for i in (0, 1):
            call(i)
    for i in (0, 1):
        assert ex.exfold_device_status(wss[i], streams[i]) == 0
        assert np.array_equal(ys[i].float().cpu().numpy(), want)
    with torch.cuda.stream(streams[0]):
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=streams[0]):
            call(0)
        ys[0].fill_(float("nan"))
        for _ in range(3):
            graph.replay()
        streams[0].synchronize()
    assert ex.exfold_device_status(wss[0], streams[0]) == 0
    assert np.array_equal(ys[0].float().cpu().numpy(), want)
