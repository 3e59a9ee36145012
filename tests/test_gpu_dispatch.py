"""Every branch of the size-dependent dispatch rules, at the sizes where each can go wrong, against the CPU oracle."""
import numpy as np
import pytest
import torch

import oracle
import synth_inputs as si
from harness import A, Case, check_decode_meta, check_output, check_prefill_meta

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,m,d", [(K, 61, 132) for K in (1, 2, 3, 4, 5, 6, 7, 8, 9, 13, 16)] + [
    (1, 1, 260), (2, 3, 2052), (2, 700, 2052), (2, 700, 2048), (3, 1, 516), (3, 3700, 260), (4, 149, 516), (4, 2400, 68), (8, 1200, 260), (8, 2, 1028)])
def test_calibration_sums_by_top_k(K, m, d):
    """Pair sums: a kernel per Top-K up to 8, tiles of four slots above (9: a ragged last tile). d = 132 leaves a tail
    after whole 128-column steps; m is not a multiple of the tokens per block; odd K: x_cal 4 bytes off a 16-byte
    boundary (fp32 calibration takes any). fp32 outputs, double sums: the oracle's
    tables to fp32 rounding of the outputs (2e-5, as in the other fp32 calibration tests). Then one token, one to a warp and one more,
    several per warp in one, two and three CTAs to an SM, rows of one column chunk, a ragged one and several, the line of K = 2."""
    N = 16
    cfg = si.LayerConfig("calk", N, 0, d, 64, K, "f32", 16, (1,), 4, (2,))
    case = Case(cfg, std=0.05, correlated=0.8)
    xc, lc = si.hidden_states(cfg, m, "x_cal"), si.router_logits(cfg, m, "logits_cal")
    ref = oracle.calibrate(A(xc), lc.numpy(), A(case.wg), A(case.wu), A(case.wd), N, K, mode=0)
    dev, ex = case.dev, case.ex
    S, L = torch.empty((N, N), device=dev), torch.empty((N, N), device=dev)
    h, lnh, n_obs = torch.empty(N, device=dev), torch.empty(N, device=dev), torch.empty((N, N), dtype=torch.int32, device=dev)
    ws = ex.alloc_workspace(case.layer, m, K)
    ws.fill_(0xFF)
    room = torch.empty(xc.numel() + 4, device=dev)
    x_dev = room[K % 2:K % 2 + xc.numel()].view(xc.shape).copy_(xc)
    rc = ex.exfold_calibrate(case.layer, x_dev, lc.to(dev), case.d_wg, case.d_wu, case.d_wd,
                             ex.make_tables(S, L, h, lnh, n_obs), ws)
    assert rc == (1 if ref["unobserved"] else 0)
    assert np.array_equal(n_obs.cpu().numpy(), ref["n_obs"])
    np.testing.assert_allclose(S.cpu().numpy(), ref["S"], rtol=2e-5, atol=2e-6)
    np.testing.assert_allclose(L.cpu().numpy(), ref["L"], rtol=1e-4, atol=2e-5)
    np.testing.assert_allclose(h.cpu().numpy(), ref["h"], rtol=1e-5)
    np.testing.assert_allclose(lnh.cpu().numpy(), ref["lnh"], rtol=1e-5, atol=1e-6)


@pytest.mark.parametrize("shape", [
    # N, shared, d, I, K, T, K', B, M
    (8, 0, 128, 256, 2, 64, 1, 16, 4),      # 8-row tiles, one row per token straight into y
    (8, 1, 132, 100, 3, 37, 2, 7, 3),       # widths off every multiple: ragged K chunks, CTAs without columns
    (4, 0, 64, 33, 2, 9, 2, 1, 4),          # I % 4 != 0: element-wise staging; slices of H past I
    (6, 1, 100, 40, 2, 300, 2, 90, 6),      # 32-row tiles with ragged last tiles, fewer slices than CTAs
    (5, 0, 256, 390, 3, 257, 3, 256, 2),    # 32-row tiles, element-wise staging, merged decode slots
    (40, 0, 36, 1100, 5, 130, 4, 33, 17),   # 16-row tiles, several feature passes per CTA
    (16, 0, 384, 640, 2, 50, 2, 40, 5),     # 8-row tiles, two feature passes
    # many tiles: 4 or 2 CTAs per cluster, of 8-, 16- and 32-row tiles, vector and element-wise
    (180, 1, 64, 96, 2, 200, 2, 109, 180),
    (90, 0, 68, 33, 3, 150, 3, 100, 90),
    (60, 0, 128, 256, 4, 500, 4, 128, 60),
    (60, 1, 36, 1100, 4, 400, 3, 70, 40),
    (8, 0, 64, 64, 2, 3000, 2, 256, 8),
    (9, 1, 132, 390, 3, 2000, 2, 256, 9),
])
def test_f32_layer_shapes(shape):
    """fp32 layers: row-tile sizes, CTAs per cluster, vector and element-wise staging, ragged widths, shared expert; routing bit-exact,
    outputs to fp32 rounding (two-level sums of at most ~1100 terms: 2e-6 of the norm; seen ~3e-7)."""
    N, ns, d, I, K, T, Kp, B, M = shape
    case = Case(si.LayerConfig("f32s", N, ns, d, I, K, "f32", T, (Kp,), B, (M,)))
    got, ref = case.run_prefill(Kp), case.oracle_prefill(Kp)
    check_prefill_meta(got, ref)
    assert check_output(got["y"], ref["y"], "f32")[1] < 2e-6
    got, ref = case.run_decode(M), case.oracle_decode(M)
    check_decode_meta(got, ref, M)
    assert check_output(got["y"], ref["y"], "f32")[1] < 2e-6


@pytest.mark.parametrize("T", [1, 31, 33, 777, 2048, 2049, 4800])
def test_routing_block_forms(T):
    """Route / scatter kernels around their block rules: one token, part blocks, token blocks shared by several blocks,
    the last call with a single super-block (2048 tokens) and the first ones with two, more blocks than SMs. Bit-exact
    permutation and offsets; every row gathered (outputs to the bf16 bound)."""
    cfg = si.LayerConfig("blocks", 40, 1, 128, 64, 5, "bf16", T, (3,), 4, (2,), logits="zipf")
    case = Case(cfg)
    got, ref = case.run_prefill(3), case.oracle_prefill(3)
    check_prefill_meta(got, ref)
    check_output(got["y"], ref["y"], "bf16")


@pytest.mark.parametrize("shape", [
    # N, shared, d, I, K, B, M
    (16, 0, 256, 384, 4, 1, 6),      # one token; a cluster of CTAs per down item
    (16, 1, 64, 64, 4, 3, 2),        # a single K chunk, shared expert, merged slots
    (40, 0, 1088, 192, 5, 8, 40),    # 17 chunks (ragged stages), full 8-column operand, pool = the batch's union
    (40, 1, 192, 320, 6, 7, 7),
    (256, 0, 128, 64, 32, 8, 200),   # largest N, K and batch
    (256, 1, 128, 64, 32, 8, 3),
    (16, 0, 2432, 128, 4, 5, 16),    # more down items than SMs: two CTAs of 8 warps
    (16, 0, 256, 384, 4, 9, 6),      # first batch of the four-kernel chain
    (16, 0, 8192, 64, 2, 8, 5),      # tokens too large for shared memory twice per SM: the chain
])
@pytest.mark.parametrize("mode", ["dynamic", "static", "router", "unaligned"])
def test_small_decode_batches(shape, mode):
    """Two-kernel decode of at most 8 tokens against the oracle: routing bit-exact, outputs to the bf16 bound. "router":
    scores from the router matrix, outputs bit-identical to the call on those scores. "unaligned": weights 16 but not 32
    bytes aligned take the chain."""
    N, ns, d, I, K, B, M = shape
    case = Case(si.LayerConfig("smalldec", N, ns, d, I, K, "bf16", 8, (1,), B, (M,)))
    ex, dev, cfg = case.ex, case.dev, case.cfg
    if mode == "unaligned":
        room = torch.empty(case.d_wg.numel() + 16, dtype=torch.bfloat16, device=dev)
        at = 8 if room.data_ptr() % 32 == 0 else 0
        case.d_wg = room[at:at + case.d_wg.numel()].view(case.d_wg.shape).copy_(case.d_wg)
        assert case.d_wg.data_ptr() % 32 == 16
    if mode == "static":
        pool = [torch.empty(M, dtype=torch.int32, device=dev), torch.empty(N, dtype=torch.int32, device=dev), torch.empty(N, device=dev)]
        sp = ex.exfold_static_pool_build(case.layer, case.tables, M, *pool)
        y = torch.full((B, d), float("nan"), dtype=torch.bfloat16, device=dev)
        ids = torch.full((B, K), -7, dtype=torch.int32, device=dev)
        w = torch.full((B, K), float("nan"), device=dev)
        ws = case.workspace(B, K)
        ex.exfold_moe_decode_static(case.layer, case.d_xd, case.d_lgd, case.d_wg, case.d_wu, case.d_wd, sp, y, ws, meta=dict(ids=ids, w=w))
        assert ex.exfold_device_status(ws) == 0
        top = oracle.decode_fold(case.lgd.numpy(), K, N, *[t.numpy() for t in case.tables_host[:3]])  # unfolded: the routes
        tgt, scl = pool[1].cpu().numpy(), pool[2].cpu().numpy()
        assert np.array_equal(ids.cpu().numpy(), tgt[top["ids"]])
        np.testing.assert_allclose(w.cpu().numpy(), top["w"] * scl[top["ids"]], rtol=1e-6, atol=1e-7)
        yr = oracle.moe_apply(A(case.xd), A(case.wg), A(case.wu), A(case.wd), tgt[top["ids"]], w.cpu().numpy(), N, ns)
        check_output(y.float().cpu().numpy(), yr, "bf16")
        return
    if mode == "router":
        wr = si.router_weights(cfg).to(dev)
        lg = torch.full((B, N), float("nan"), device=dev)
        y = torch.full((B, d), float("nan"), dtype=torch.bfloat16, device=dev)
        ws = case.workspace(B, K)
        ex.exfold_moe_decode_layer(case.layer, case.d_xd, wr, case.d_wg, case.d_wu, case.d_wd, case.tables, M, y, ws, lg)
        assert ex.exfold_device_status(ws) == 0
        case.d_lgd = lg
        case.lgd = lg.cpu()
    got, ref = case.run_decode(M), case.oracle_decode(M)
    check_decode_meta(got, ref, M)
    check_output(got["y"], ref["y"], "bf16")
    if mode == "router":
        assert np.array_equal(got["y"], y.float().cpu().numpy())
    plain = case.run_decode(M, with_meta=False)  # without metadata only the batch's experts get targets
    assert np.array_equal(got["y"], plain["y"])


@pytest.mark.parametrize("B", [80, 81, 87, 96, 97, 103, 128])
@pytest.mark.parametrize("N", [31, 32, 64, 65, 100, 256])
def test_decode_router_scores_by_batch(B, N):
    """Router scores inside the decode call, a token per cluster (a warp takes one expert, above 64 experts two) or eight
    (from 97 tokens and 65 experts on; ragged last cluster, experts not a multiple of the tiles): the bits of
    exfold_router_logits."""
    case = Case(si.LayerConfig("rt", N, 0, 320, 64, 4, "bf16", 8, (1,), B, (6,)))
    ex, dev = case.ex, case.dev
    wr = si.router_weights(case.cfg).to(dev)
    lg, want = torch.full((B, N), float("nan"), device=dev), torch.full((B, N), float("nan"), device=dev)
    y = torch.empty((B, 320), dtype=torch.bfloat16, device=dev)
    ws = case.workspace(B, 4)
    ex.exfold_moe_decode_layer(case.layer, case.d_xd, wr, case.d_wg, case.d_wu, case.d_wd, case.tables, 6, y, ws, lg)
    assert ex.exfold_device_status(ws) == 0
    ex.exfold_router_logits(case.layer, case.d_xd, wr, want, ws)
    assert torch.equal(lg, want)
    case.lgd, case.d_lgd = lg.cpu(), lg
    ref = case.oracle_decode(6)
    check_output(y.float().cpu().numpy(), ref["y"], "bf16")


@pytest.mark.parametrize("B", [1, 9, 80, 81, 128, 129, 256])
@pytest.mark.parametrize("N", [5, 40, 256])
def test_decode_router_scores_of_short_rows(B, N):
    """Rows of 64: the shortest dot products, whose scores the cluster's CTAs write to the first one soonest after its
    start; CTAs and warps without experts. Against double sums (the bound of test_router_scores_by_prompt_length), the
    call on them against the oracle, the same bits every time."""
    d, K = 64, 4
    case = Case(si.LayerConfig("short", N, 0, d, 64, K, "bf16", 8, (1,), B, (3,)))
    ex, dev = case.ex, case.dev
    wr = si.router_weights(case.cfg).to(dev)
    x64, w64 = case.d_xd.double(), wr.double()
    want, bound = x64 @ w64.T, d * 2.0 ** -23 * (x64.abs() @ w64.abs().T)
    y, first = torch.empty((B, d), dtype=torch.bfloat16, device=dev), None
    ws = case.workspace(B, K)
    for _ in range(20):
        lg = torch.full((B, N), float("nan"), device=dev)
        ex.exfold_moe_decode_layer(case.layer, case.d_xd, wr, case.d_wg, case.d_wu, case.d_wd, case.tables, 3, y, ws, lg)
        got = (lg, y.clone())
        first = first or got
        assert torch.equal(got[0], first[0]) and torch.equal(got[1], first[1])
    assert ex.exfold_device_status(ws) == 0
    assert bool(((first[0].double() - want).abs() <= bound).all())
    case.lgd, case.d_lgd = first[0].cpu(), first[0]
    check_output(first[1].float().cpu().numpy(), case.oracle_decode(3)["y"], "bf16")


@pytest.mark.parametrize("rows,ns,d,I", [
    ([1, 3, 4, 5, 63, 64, 65, 51], 0, 256, 384),     # 256 tokens: gathered up to 64 rows, dense above
    ([64, 65], 1, 64, 64),                           # 129 tokens, one K chunk, half-width items, the shared expert dense
    ([64, 64, 1], 0, 1088, 192),                     # every group gathered, 17 chunks
    ([130, 126], 0, 128, 192),                       # none
    ([2] * 100, 0, 128, 128),                        # many small groups
    # the lists above leave SMs idle (the last aside), so that few rows or none are gathered; these fill them, or nearly
    ([1, 3, 4, 5, 63, 64, 65, 51], 0, 256, 2432),
    ([64, 65], 1, 64, 6336),
    ([64, 64, 1], 0, 1088, 6336),
    ([42, 43, 41] + [3] * 37, 0, 128, 384),          # 120 of 148 SMs: up to 42 rows
])
@pytest.mark.parametrize("place", ["mixed", "sorted"])
def test_decode_group_sizes_above_128_tokens(rows, ns, d, I, place):
    """More than 128 tokens: the gate/up items of small groups gather their rows, larger groups run per token tile. Each
    token's one expert is given; "sorted" puts a group's tokens next to one another (a group then touches one tile or two)."""
    B, N = sum(rows), len(rows)
    case = Case(si.LayerConfig("groups", N, ns, d, I, 1, "bf16", 8, (1,), B, (N,)))
    owner = np.repeat(np.arange(N), rows)
    if place == "mixed":
        owner = np.random.default_rng(5).permutation(owner)
    case.lgd[torch.arange(B), torch.from_numpy(owner)] = 20.0
    case.d_lgd = case.lgd.to(case.dev)
    got, ref = case.run_decode(N), case.oracle_decode(N)
    check_decode_meta(got, ref, N)
    assert np.array_equal(got["ids"].reshape(-1), owner)
    check_output(got["y"], ref["y"], "bf16")
    plain = case.run_decode(N, with_meta=False)
    assert np.array_equal(got["y"], plain["y"])


@pytest.mark.parametrize("B,N,K,M", [
    (9, 16, 5, 4),       # slots not a multiple of four, more members than pool places
    (33, 40, 3, 40),     # the pool is the batch's union
    (129, 40, 3, 16),    # two token tiles, ragged
    (64, 256, 8, 200),   # more candidates than one round trip holds
    (256, 128, 16, 70),  # the most slots
    (256, 130, 8, 1),
])
@pytest.mark.parametrize("h_step", [0.0, 2.0 ** -23])
def test_decode_pool_of_near_ties(B, N, K, M, h_step):
    """Experts in pairs of equal router scores and (almost) equal norms: pool scores that agree in their upper halves (equal,
    or apart by one unit of the norm's last place) are ranked by the whole score, then by id."""
    case = Case(si.LayerConfig("ties", N, 0, 64, 64, K, "bf16", 8, (1,), B, (M,)))
    case.lgd[:, 1::2] = case.lgd[:, 0:N - N % 2:2]
    case.d_lgd = case.lgd.to(case.dev)
    S, L, h, lnh = case.tables_host
    h = 1.0 + h_step * (torch.arange(N) % 2).to(h.dtype)
    case.set_tables((S, L, h, torch.log(h)))
    got, ref = case.run_decode(M), case.oracle_decode(M)
    check_decode_meta(got, ref, M)
    check_output(got["y"], ref["y"], "bf16")
    plain = case.run_decode(M, with_meta=False)
    assert np.array_equal(got["y"], plain["y"])


@pytest.mark.parametrize("I,M,ns,d", [(2368, 2, 0, 320), (2368, 2, 1, 320), (384, 12, 0, 320), (384, 12, 1, 320), (384, 13, 0, 320),
                                      (64, 1, 0, 64), (832, 5, 0, 320), (448, 5, 0, 1088), (512, 5, 1, 1088)])
@pytest.mark.parametrize("B", [20, 100, 140])
def test_decode_slice_widths(B, I, M, ns, d):
    """Few groups: 32-wide gate/up slices up to one per SM (148 = 2 x 2368 / 32, 144 = 12 x 384 / 32), wider ones beyond; 64 or
    128 output columns per down tile (hidden sizes that leave the last tile short), with and without the K split."""
    case = Case(si.LayerConfig("slices", 16, ns, d, I, 3, "bf16", 8, (1,), B, (M,)))
    got, ref = case.run_decode(M), case.oracle_decode(M)
    check_decode_meta(got, ref, M)
    check_output(got["y"], ref["y"], "bf16")


@pytest.mark.parametrize("T", [1, 5, 128, 129, 300, 777, 5000])
@pytest.mark.parametrize("N,d", [(31, 64), (40, 320), (130, 2048), (256, 1088)])
def test_router_scores_by_prompt_length(T, N, d):
    """Dot-product kernel up to one row tile (one or 4 x 4 scores per warp), tensor cores with K split over a cluster above
    (one, two and eight parts, ragged last tile, experts off every multiple) against double sums. Products of bf16 are
    exact in fp32, so the error is the additions': at most d of them, each within 2^-23 of the partial sum's bound
    sum |w x|."""
    from paper_2608_24938_b200 import binding as ex
    dev = torch.device("cuda:0")
    g = torch.Generator(device=dev)
    g.manual_seed(T + N)
    x = torch.randn((T, d), generator=g, device=dev).to(torch.bfloat16)
    wr = (torch.randn((N, d), generator=g, device=dev) * d ** -0.5).to(torch.bfloat16)
    layer = ex.make_layer(N, 0, d, 64, 2, "bf16")
    ws = ex.alloc_workspace(layer, T, 1)
    ws.fill_(0xFF)  # also a status record to clear
    lg = torch.full((T, N), float("nan"), device=dev)
    assert ex.exfold_router_logits(layer, x, wr, lg, ws) == 0
    assert ex.exfold_device_status(ws) == 0
    want = x.double() @ wr.double().T
    bound = d * 2.0 ** -23 * (x.double().abs() @ wr.double().abs().T)
    assert bool(((lg.double() - want).abs() <= bound).all())


@pytest.mark.parametrize("Kp,ns,d", [(1, 1, 64), (2, 0, 192), (3, 1, 4160), (5, 0, 256), (7, 0, 320), (8, 0, 128), (8, 1, 128),
                                     (9, 0, 64), (10, 1, 128)])
def test_rows_summed_per_token(Kp, ns, d):
    """The per-token sum by number of rows (2 to 9 known at compile time, more in batches of eight) and widths that leave
    part of a block idle or take two passes."""
    cfg = si.LayerConfig("sum", 16, ns, d, 64, 10, "bf16", 70, (Kp,), 4, (2,))
    case = Case(cfg)
    got, ref = case.run_prefill(Kp), case.oracle_prefill(Kp)
    check_prefill_meta(got, ref)
    check_output(got["y"], ref["y"], "bf16")


@pytest.mark.parametrize("T", [1, 3, 8, 9])
@pytest.mark.parametrize("N,ns,d,I,K,Kp", [(16, 0, 256, 384, 4, 2), (40, 1, 1088, 192, 6, 6), (256, 1, 128, 64, 32, 32),
                                            (8, 0, 2432, 128, 2, 1)])
def test_few_token_prefill(T, N, ns, d, I, K, Kp):
    """Prefill of at most 8 tokens on the small-batch kernels (9: the grouped GEMMs): metadata bit-exact, outputs to the bf16
    bound and the same bits with metadata, without, and for every gemm_path."""
    case = Case(si.LayerConfig("few", N, ns, d, I, K, "bf16", T, (Kp,), 4, (2,)))
    got, ref = case.run_prefill(Kp), case.oracle_prefill(Kp)
    check_prefill_meta(got, ref)
    check_output(got["y"], ref["y"], "bf16")
    for path in (0, 1, 2):
        assert np.array_equal(got["y"], case.run_prefill(Kp, with_meta=False, gemm_path=path)["y"])


@pytest.mark.parametrize("T", [4095, 4097, 6145, 8192, 8193])
def test_host_prefill_covers_every_token(T):
    """Chunked host-buffer prefill around multiples of its chunks (8193 = four chunks of 2048 and one token more): every
    token computed, bit-identical to the device call."""
    cfg = si.LayerConfig("chunk", 8, 0, 64, 64, 2, "bf16", T, (1,), 4, (2,))
    case = Case(cfg)
    want = case.run_prefill(1, with_meta=False)["y"]
    ex = case.ex
    ws = ex.alloc_workspace(case.layer, T, 1, host_staging=True)
    y = torch.full((T, 64), float("nan"), dtype=torch.bfloat16).pin_memory()
    ex.exfold_moe_prefill_host(case.layer, case.x.pin_memory(), case.lg.pin_memory(), case.d_wg, case.d_wu, case.d_wd, case.tables, 1, y, ws)
    assert ex.exfold_device_status(ws) == 0
    assert np.array_equal(y.float().numpy(), want)


@pytest.mark.parametrize("T,N,ns,d,I,K,Kp", [
    (1, 8, 0, 128, 256, 2, 1), (7, 8, 1, 128, 256, 2, 2), (64, 8, 0, 128, 256, 2, 1), (65, 8, 0, 128, 250, 2, 2), (128, 8, 0, 64, 96, 3, 1),
    (127, 16, 0, 64, 96, 4, 2), (129, 16, 0, 64, 96, 4, 1), (9, 33, 1, 132, 64, 5, 3), (20, 128, 0, 64, 64, 8, 2), (16, 2, 0, 64, 64, 2, 1),
    (3, 100, 1, 96, 64, 32, 16), (20, 129, 0, 64, 64, 3, 1), (2, 8, 0, 3584, 3584, 2, 2)])
def test_fp32_prefill_that_routes_in_its_ffn_kernel(T, N, ns, d, I, K, Kp):
    """Few tokens of an fp32 layer: routing inside the FFN kernel (up to 128 tokens, 128 experts, one wave of clusters) and the
    kernels of its own beyond; metadata bit-exact, outputs to fp32 rounding."""
    case = Case(si.LayerConfig("f32r", N, ns, d, I, K, "f32", T, (Kp,), 4, (2,)))
    got, ref = case.run_prefill(Kp), case.oracle_prefill(Kp)
    check_prefill_meta(got, ref)
    assert check_output(got["y"], ref["y"], "f32")[1] < 2e-6
    assert np.array_equal(got["y"], case.run_prefill(Kp, with_meta=False)["y"])


@pytest.mark.parametrize("T,ns,d,I,launches", [(93, 1, 1600, 1024, 2), (93, 1, 2048, 1536, 4), (60, 0, 2048, 1536, 1), (20, 1, 2048, 1536, 2)])
def test_fp32_routing_where_a_wave_holds_the_tiles(T, ns, d, I, launches):
    """The FFN kernel routes only where all its clusters run at once: two CTAs to an SM up to 3130 to 3500 of d + I, one above, where
    its routing state does not fit twice. One launch (rows stored into y) or two, else four."""
    case = Case(si.LayerConfig("f32w", 8, ns, d, I, 2, "f32", T, (1,), 4, (2,)))
    before = case.ex.exfold_launch_count()
    got = case.run_prefill(1)
    assert case.ex.exfold_launch_count() - before == launches
    idx = np.arange(0, T, 7)
    ref = case.oracle_prefill(1, tok_idx=idx)
    check_prefill_meta(got, ref)
    assert check_output(got["y"][idx], ref["y"], "f32")[1] < 2e-6


@pytest.mark.parametrize("thr,rescale,conf", [(0.6, False, False), (0.6, True, False), (float("inf"), False, True), (0.5, True, True), (-1.0, True, False)])
@pytest.mark.parametrize("dtype,T,N,K,Kp", [("f32", 64, 8, 4, 2), ("f32", 128, 40, 4, 3), ("f32", 150, 8, 4, 2), ("bf16", 1, 16, 6, 3), ("bf16", 8, 40, 6, 2)])
def test_safeguards_where_the_ffn_kernels_route(dtype, T, N, K, Kp, thr, rescale, conf):
    """Loss threshold, rescale and confidence split of the calls whose FFN kernel routes its tokens itself (fp32 up to 128 tokens, and
    150 beside it; bf16 up to 8 without metadata): metadata as the oracle's, the same bits without it."""
    d = 128
    case = Case(si.LayerConfig("safe", N, 1, d, 192, K, dtype, T, (Kp,), 4, (2,)))
    ex, dev = case.ex, case.dev
    S, L, h, lnh = case.np_tables()
    ref = oracle.prefill_fold_safe(case.lg.numpy(), K, Kp, S, L, lnh, loss_thr=thr, rescale=rescale, confidence=conf)
    yref = oracle.moe_apply(A(case.x), A(case.wg), A(case.wu), A(case.wd), ref["ids"], ref["w"], N, 1)
    i32 = dict(dtype=torch.int32, device=dev)
    meta = dict(ids=torch.full((T, Kp), -7, **i32), w=torch.full((T, Kp), float("nan"), device=dev),
                omit_src=torch.full((T, K - Kp), -7, **i32), omit_tgt=torch.full((T, K - Kp), -7, **i32))
    ys = []
    for m in (meta, None):
        ws, y = case.workspace(T, Kp), torch.full((T, d), float("nan"), dtype=case.d_wg.dtype, device=dev)
        ex.exfold_moe_prefill_ex(case.layer, case.d_x, case.d_lg, case.d_wg, case.d_wu, case.d_wd, case.tables, Kp, y, ws,
                                 loss_threshold=thr, rescale=rescale, confidence_split=conf, meta=m)
        assert ex.exfold_device_status(ws) == 0
        ys.append(y.float().cpu().numpy())
    for k in ("ids", "omit_src", "omit_tgt"):
        assert np.array_equal(meta[k].cpu().numpy(), ref[k]), k
    np.testing.assert_allclose(meta["w"].cpu().numpy(), ref["w"], rtol=2e-5, atol=2e-5)  # as in test_prefill_safeguards
    check_output(ys[0], yref, dtype)
    assert np.array_equal(ys[0], ys[1])


@pytest.mark.parametrize("T,B,N,ns,d,I,K,Kp,M", [(456, 116, 8, 0, 128, 256, 2, 2, 3), (600, 230, 8, 0, 64, 96, 2, 2, 2), (700, 33, 7, 1, 68, 90, 5, 5, 1)])
def test_fp32_short_tiles_of_long_groups(T, B, N, ns, d, I, K, Kp, M):
    """Groups of many short tiles (a few waves of clusters, four or two CTAs each) and, last, the tall tiles beyond."""
    case = Case(si.LayerConfig("f32t", N, ns, d, I, K, "f32", T, (Kp,), B, (M,)))
    got, ref = case.run_prefill(Kp), case.oracle_prefill(Kp)
    check_prefill_meta(got, ref)
    assert check_output(got["y"], ref["y"], "f32")[1] < 2e-6
    got, ref = case.run_decode(M), case.oracle_decode(M)
    check_decode_meta(got, ref, M)
    assert check_output(got["y"], ref["y"], "f32")[1] < 2e-6


@pytest.mark.parametrize("B,N,ns,d,I,K,M", [
    (1, 8, 0, 128, 256, 2, 2), (16, 8, 0, 128, 256, 2, 4), (31, 8, 1, 128, 250, 2, 8), (32, 8, 0, 64, 96, 3, 1), (33, 16, 0, 64, 96, 4, 6),
    (64, 33, 0, 132, 64, 5, 3), (128, 8, 0, 64, 64, 2, 2), (129, 8, 0, 64, 64, 2, 2), (9, 128, 1, 64, 64, 9, 100), (9, 129, 0, 64, 64, 4, 5),
    (16, 40, 0, 64, 64, 32, 7)])
def test_fp32_decode_that_routes_in_its_ffn_kernel(B, N, ns, d, I, K, M):
    """Few tokens of an fp32 layer: pool, targets and lists inside the FFN kernel (up to 128 tokens, 128 experts, one wave of
    clusters) and the kernels of its own beyond, dynamic and static pool: metadata bit-exact, outputs to fp32 rounding."""
    case = Case(si.LayerConfig("f32d", N, ns, d, I, K, "f32", 8, (1,), B, (M,)))
    got, ref = case.run_decode(M), case.oracle_decode(M)
    check_decode_meta(got, ref, M)
    assert check_output(got["y"], ref["y"], "f32")[1] < 2e-6
    ex, dev = case.ex, case.dev
    pool_ids, target = torch.empty(M, dtype=torch.int32, device=dev), torch.empty(N, dtype=torch.int32, device=dev)
    scale = torch.empty(N, device=dev)
    pool = ex.exfold_static_pool_build(case.layer, case.tables, M, pool_ids, target, scale)
    ws, y = case.workspace(B, K), torch.full((B, d), float("nan"), device=dev)
    ids = torch.empty((B, K), dtype=torch.int32, device=dev)
    w = torch.empty((B, K), device=dev)
    ex.exfold_moe_decode_static(case.layer, case.d_xd, case.d_lgd, case.d_wg, case.d_wu, case.d_wd, pool, y, ws, meta=dict(ids=ids, w=w))
    assert ex.exfold_device_status(ws) == 0
    routed = case.lgd.topk(K, dim=1).indices
    assert np.array_equal(ids.cpu().numpy(), target.cpu().numpy()[routed.numpy()])
    yr = oracle.moe_apply(A(case.xd), A(case.wg), A(case.wu), A(case.wd), ids.cpu().numpy(), w.cpu().numpy(), N, ns)
    assert check_output(y.cpu().numpy(), yr, "f32")[1] < 2e-6
