"""Kernel parity on the GPU: every kernel of the path, called through the C ABI, against the CPU oracle
on the same seeded inputs; sizes span several tiles and ragged tails, plus the degenerate cases."""
import json
from dataclasses import replace

import numpy as np
import pytest

import seeded_inputs as si

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle.forward import OracleModel, bf16_round  # noqa: E402
from paper_2609_06172_b200 import binding as tb  # noqa: E402
from paper_2609_06172_b200.session import model_cfg  # noqa: E402

DEV = "cuda:0"
KCFG = si.ModelConfig("k", L=1, d=128, Hq=4, Hkv=2, Dh=64, F=256, V=512, B=2, S=8, T=8, TK=4, seed=7, budget_rule="half_w")


def bf16_dev(bits):
    return torch.from_numpy(bits.view(np.int16)).to(DEV).view(torch.bfloat16)


def rnd_bits(role, n):
    return si.normal_bf16_bits(1234, role, 0, n)


def kernels_of(call, tmp_path):
    """Names and launch records ("shared memory": static and dynamic, bytes; "grid") of the kernels a call launches, in order."""
    call()                                                 # (function attributes, first-use allocations)
    torch.cuda.synchronize()
    with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as prof:
        call()
        torch.cuda.synchronize()
    path = tmp_path / "trace.json"
    prof.export_chrome_trace(str(path))
    events = [e for e in json.loads(path.read_text())["traceEvents"] if e.get("cat") == "kernel"]
    return [(e["name"], e["args"]) for e in sorted(events, key=lambda e: e["ts"])]


def oracle():
    lay = si.build_layout(KCFG)
    return OracleModel(KCFG, si.weights_as_bits(lay))


def bf16_close(got_f32, want_f32, frac=0.01):
    """Equal up to one bf16 ulp, and different at all in at most `frac` of the entries (rounding flips
    where fp32 summation order differs by a last bit)."""
    got, want = np.asarray(got_f32, np.float32), np.asarray(want_f32, np.float32)
    tol = np.maximum(np.abs(want), 1e-30) * 2.0 ** -7
    assert (np.abs(got - want) <= tol).all(), float(np.abs(got - want).max())
    assert (got != want).mean() <= frac


@pytest.mark.parametrize("M,n,K", [(1, 300, 256), (1, 4096, 2048), (2, 129, 64), (3, 1000, 512), (8, 1030, 512),
                                   (13, 77, 128), (16, 260, 1024), (17, 64, 96), (33, 130, 96), (200, 260, 1024),
                                   (64, 64, 32), (1, 1, 8), (70, 5, 8), (129, 257, 72), (300, 520, 1096), (512, 2048, 2048),
                                   (1000, 136, 8192),
                                   # few rows, long K at M <= 2: the split-K GEMV (two rows per CTA; one row per CTA up to 1024 rows),
                                   # odd row counts, K not a multiple of the 256-element chunk, more CTAs than resident slots
                                   (1, 2048, 8192), (2, 2051, 8200), (1, 513, 8192), (2, 1, 16384), (1, 4735, 8192),
                                   # 33 - 64 activation rows on blocks of few rows: one 128-row weight tile per CTA, K in two or four slices
                                   (33, 1030, 512), (48, 2049, 4096), (64, 130, 96), (40, 4090, 64),
                                   # ... and on blocks of many rows
                                   (40, 4720, 64), (64, 4096, 1032), (20, 8200, 128)])
@pytest.mark.parametrize("accumulate", [0, 1])
def test_gemm_matches_oracle(M, n, K, accumulate):
    a_bits, w_bits = rnd_bits(1, M * K).reshape(M, K), rnd_bits(2, n * K).reshape(n, K)
    A, W = bf16_dev(a_bits), bf16_dev(w_bits)
    ldc, col0 = n + 24, 8
    c0 = np.random.default_rng(M * n).standard_normal((M, ldc)).astype(np.float32) * 0.01
    Cd = torch.from_numpy(c0.copy()).to(DEV)
    tb.k_gemm(A, W, Cd, M, n, K, ldc, col0, accumulate)
    torch.cuda.synchronize()
    got = Cd.cpu().numpy()
    o = oracle()
    want = o.linear(si.bf16_bits_to_f32(a_bits), si.bf16_bits_to_f32(w_bits).astype(np.float64)).astype(np.float64)
    exp = c0.astype(np.float64).copy()
    exp[:, col0:col0 + n] = want + (c0[:, col0:col0 + n] if accumulate else 0)
    scale = np.abs(want).max() + 1e-6
    assert np.abs(got - exp).max() < 2e-5 * max(scale, 0.01) + 1e-7
    assert np.array_equal(got[:, :col0], c0[:, :col0]) and np.array_equal(got[:, col0 + n:], c0[:, col0 + n:])


def test_tensor_core_gemm_agrees_with_cuda_core_gemm_and_reports_no_timeout():
    """Same inputs through both M > 16 kernels: the tcgen05 path and the CUDA-core tiles (an on-device cross-check
    besides the oracle), then the tensor-core kernel's bounded-wait error word must still be zero."""
    M, n, K = 640, 1408, 2048
    A, W = bf16_dev(rnd_bits(5, M * K).reshape(M, K)), bf16_dev(rnd_bits(6, n * K).reshape(n, K))
    outs = []
    for impl in (0, 1):
        tb.k_gemm_select(impl)
        Cd = torch.zeros(M, n, dtype=torch.float32, device=DEV)
        tb.k_gemm(A, W, Cd, M, n, K, n, 0, 0)
        torch.cuda.synchronize()
        outs.append(Cd.cpu().numpy())
    tb.k_gemm_select(0)
    assert np.abs(outs[0] - outs[1]).max() < 2e-5 * np.abs(outs[1]).max()
    assert np.abs(outs[0]).max() > 0
    assert tb.k_gemm_status() == 0


@pytest.mark.parametrize("M,n,K,acc", [(300, 520, 1096, 0), (129, 257, 72, 1), (1024, 1536, 512, 0), (640, 2300, 2048, 1), (4096, 4096, 256, 0)])
def test_persistent_tensor_core_gemm_matches_per_tile_kernel_and_oracle(M, n, K, acc):
    """The paired 256x256 kernel and the persistent 128x256 kernel (forced, even on small problems: ragged tiles, a pair
    whose second CTA has no valid row, fewer tiles than SMs, several tiles per CTA) against the per-tile kernel and the
    oracle."""
    a_bits, w_bits = rnd_bits(11, M * K).reshape(M, K), rnd_bits(12, n * K).reshape(n, K)
    A, W = bf16_dev(a_bits), bf16_dev(w_bits)
    c0 = np.random.default_rng(7).standard_normal((M, n)).astype(np.float32) * 0.01
    outs = []
    for variant in (3, 2, 1):
        tb.k_gemm_tc_variant(variant)
        Cd = torch.from_numpy(c0.copy()).to(DEV)
        tb.k_gemm(A, W, Cd, M, n, K, n, 0, acc)
        torch.cuda.synchronize()
        outs.append(Cd.cpu().numpy())
    tb.k_gemm_tc_variant(0)
    assert tb.k_gemm_status() == 0
    want = oracle().linear(si.bf16_bits_to_f32(a_bits), si.bf16_bits_to_f32(w_bits).astype(np.float64)).astype(np.float64) + (c0 if acc else 0)
    scale = np.abs(want).max()
    for o in outs:
        assert np.abs(o - want).max() < 2e-5 * scale + 1e-7
    assert np.abs(outs[0] - outs[2]).max() < 2e-5 * scale + 1e-7 and np.abs(outs[1] - outs[2]).max() < 2e-5 * scale + 1e-7


@pytest.mark.parametrize("M,n,K,acc", [(17, 300, 264, 0), (32, 4100, 1024, 1), (33, 1030, 512, 1), (64, 130, 96, 0), (65, 2049, 1024, 1),
                                       (128, 4096, 512, 0), (100, 129, 72, 1), (48, 8200, 256, 0)])
def test_tensor_core_gemm_with_the_weights_as_the_128_row_operand(M, n, K, acc):
    """Up to 128 activation rows: the per-tile kernel with its operands swapped (tile rows are weight rows, the tile is
    stored transposed), forced, against the oracle; ragged weight tiles, ragged token counts, a column offset."""
    a_bits, w_bits = rnd_bits(13, M * K).reshape(M, K), rnd_bits(14, n * K).reshape(n, K)
    A, W = bf16_dev(a_bits), bf16_dev(w_bits)
    ldc, col0 = n + 12, 4
    c0 = np.random.default_rng(9).standard_normal((M, ldc)).astype(np.float32) * 0.01
    tb.k_gemm_tc_variant(4)
    Cd = torch.from_numpy(c0.copy()).to(DEV)
    tb.k_gemm(A, W, Cd, M, n, K, ldc, col0, acc)
    torch.cuda.synchronize()
    tb.k_gemm_tc_variant(0)
    assert tb.k_gemm_status() == 0
    got = Cd.cpu().numpy()
    want = oracle().linear(si.bf16_bits_to_f32(a_bits), si.bf16_bits_to_f32(w_bits).astype(np.float64)).astype(np.float64)
    exp = c0.astype(np.float64).copy()
    exp[:, col0:col0 + n] = want + (c0[:, col0:col0 + n] if acc else 0)
    assert np.abs(got - exp).max() < 2e-5 * max(np.abs(want).max(), 0.01) + 1e-7
    assert np.array_equal(got[:, :col0], c0[:, :col0]) and np.array_equal(got[:, col0 + n:], c0[:, col0 + n:])


# (M, K, n, residual): the weight-block products of the prefill steps the benchmark times - M = B * S of the 8B shape (8 x 1024),
# the MoE shape (32 x 512) and the 70B shape (16 x 2048); K = d or FFN; n = rows of one 32 MiB sub-range block of that matrix
REAL_PREFILL = [(8192, 4096, 4096, 0), (8192, 14336, 1152, 1), (16384, 4096, 4096, 0), (32768, 8192, 2048, 0), (32768, 28672, 512, 1)]


@pytest.mark.parametrize("M,K,n,acc", REAL_PREFILL)
def test_gemm_at_the_real_prefill_shapes_sampled_rows_against_the_oracle(M, K, n, acc):
    """Full-size prefill products in the launch configuration the benchmark times (automatic kernel choice: the paired
    tcgen05 kernel).  A full CPU product would take minutes, and an output row depends on one activation row only, so
    the oracle recomputes 64 sampled rows - first, last, the rows around every 128- and 256-row tile edge it can hit,
    and seeded random ones - from the same bf16 inputs, in double.  The rows in between are covered by a checksum
    property that holds at any size: the column sums of C equal (column sums of A) . W^T."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(M * 31 + K)
    A = torch.randn((M, K), device=DEV, generator=gen).bfloat16()
    W = (torch.randn((n, K), device=DEV, generator=gen) * 0.02).bfloat16()
    c0 = (torch.randn((M, n), device=DEV, generator=gen) * 0.5).float() if acc else None
    Cd = c0.clone() if acc else torch.empty((M, n), dtype=torch.float32, device=DEV)
    tb.k_gemm(A, W, Cd, M, n, K, n, 0, acc)
    torch.cuda.synchronize()
    assert tb.k_gemm_status() == 0
    rng = np.random.default_rng(M + K)
    rows = sorted(set([0, 1, 127, 128, 255, 256, M // 2 - 1, M // 2, M - 257, M - 256, M - 129, M - 128, M - 2, M - 1] + rng.integers(0, M, 50).tolist()))[:64]
    ridx = torch.tensor(rows, device=DEV)
    a_rows = si.bf16_bits_to_f32(A[ridx].view(torch.int16).cpu().numpy().view(np.uint16))
    w_bits = W.view(torch.int16).cpu().numpy().view(np.uint16)
    want = oracle().linear(a_rows, si.bf16_bits_to_f32(w_bits).astype(np.float64)).astype(np.float64)
    if acc:
        want = want + c0[ridx].cpu().numpy().astype(np.float64)
    got = Cd[ridx].cpu().numpy().astype(np.float64)
    scale = np.abs(want).max()
    # 2e-5 of the largest output holds up to K = 8192 (every other GEMM test).  The tensor cores add each 16-deep partial
    # product into the fp32 accumulator without round-to-nearest, so the error has a part that grows linearly with the
    # K / 16 accumulation steps (bound: K / 16 * 2^-23 = 2.1e-4 at K = 28672; measured 3.2e-5): the tolerance grows with K
    tol = 2e-5 * max(1.0, K / 8192)
    assert np.abs(got - want).max() < tol * scale + 1e-7, (np.abs(got - want).max(), scale)
    # every row, through a property: sum_m C[m, j] = (sum_m A[m, :]) . W[j, :]  (+ sum_m C0[m, j]), in double
    colsum = Cd.double().sum(dim=0).cpu().numpy()
    asum = A.double().sum(dim=0).cpu().numpy()
    ref = si.bf16_bits_to_f32(w_bits).astype(np.float64) @ asum + (c0.double().sum(dim=0).cpu().numpy() if acc else 0.0)
    # fp32 accumulation error of one output element is ~1e-6 of its scale; M of them add up at random
    # (the accumulator's rounding bias has one sign per column, so over M rows it adds up linearly in the worst case)
    assert np.abs(colsum - ref).max() < tol * scale * M * 0.25 + 1e-6, (np.abs(colsum - ref).max(), scale)
    # and no element is non-finite or left unwritten
    assert bool(torch.isfinite(Cd).all())


@pytest.mark.parametrize("variant,M,n,K", [(1, 256, 256, 512), (2, 384, 512, 512), (3, 512, 512, 1024)])
def test_tensor_core_gemm_gives_up_on_a_wait_that_runs_out_and_recovers(variant, M, n, K):
    """Failure detection without a fault: with the wait limit set to 2 ms and the TMA thread of the first CTA (pair)
    leaving out its second load step, the MMA thread's wait for that stage runs out.  The kernel must return by itself,
    the error word must name the wait (role 2 = MMA issuer), the CTA that gave up must have stored nothing, every other
    CTA's tile must be right, and - limits restored, error word cleared - the next launch must be correct again."""
    a_bits, w_bits = rnd_bits(51, M * K).reshape(M, K), rnd_bits(52, n * K).reshape(n, K)
    A, W = bf16_dev(a_bits), bf16_dev(w_bits)
    want = oracle().linear(si.bf16_bits_to_f32(a_bits), si.bf16_bits_to_f32(w_bits).astype(np.float64)).astype(np.float64)
    SENT = 12345.0
    tb.k_status_clear()
    tb.k_gemm_tc_variant(variant)
    try:
        tb.k_wait_test(2_000_000, 1)
        Cd = torch.full((M, n), SENT, dtype=torch.float32, device=DEV)
        tb.k_gemm(A, W, Cd, M, n, K, n, 0, 0)
        torch.cuda.synchronize()                              # returns: nothing hangs, nothing faults
        code = tb.k_gemm_status()
        assert code >> 8 == 2, hex(code)                      # the MMA issuer's wait for a stage ran out first
        got = Cd.cpu().numpy()
        untouched = got == SENT
        rows, cols = (256, 256) if variant == 3 else (128, 256 if variant == 2 else 128)
        assert untouched[:rows, :cols].all()                  # the first CTA (pair) owns the first tile: nothing stored
        done = ~untouched
        assert done.sum() == M * n - rows * cols              # every other tile was stored, and correctly
        assert np.abs(got[done] - want[done]).max() < 2e-5 * np.abs(want).max() + 1e-7
    finally:
        tb.k_wait_test(0, -1)
        tb.k_status_clear()
    Cd = torch.zeros((M, n), dtype=torch.float32, device=DEV)
    tb.k_gemm(A, W, Cd, M, n, K, n, 0, 0)
    torch.cuda.synchronize()
    tb.k_gemm_tc_variant(0)
    assert tb.k_gemm_status() == 0
    assert np.abs(Cd.cpu().numpy() - want).max() < 2e-5 * np.abs(want).max() + 1e-7


@pytest.mark.parametrize("Dh", [64, 128])
def test_tensor_core_attention_gives_up_on_a_wait_that_runs_out_and_recovers(Dh):
    """The same for the tcgen05 attention kernel: the first CTA's TMA thread never requests its second V block, the
    roles that depend on it - the P V issuer (code 3: a K/V load), the softmax warps (1: S, 2: P V), the S issuer - all
    start waiting within microseconds of each other and the first whose 2 ms run out records its code; that CTA stores
    nothing, the others finish, and the next launch is correct."""
    cfg = replace(KCFG, Dh=Dh, Hq=4, Hkv=2, TK=64, S=256, T=0, B=2, d=4 * Dh)
    mc = model_cfg(cfg)
    B, S = cfg.B, cfg.S
    kt, vt = make_tiles(cfg, B)
    for j, (k, v) in enumerate(zip(kt, vt)):
        k.copy_(bf16_dev(rnd_bits(60 + j, k.numel())) * 30)
        v.copy_(bf16_dev(rnd_bits(70 + j, v.numel())) * 30)
    qb = (bf16_dev(rnd_bits(80, B * S * cfg.Hq * Dh)) * 30).view(B * S, cfg.Hq * Dh)
    o = OracleModel(cfg, {})
    o.K[0], o.V[0] = tiles_to_cache(kt, cfg, B)[:, :, :S], tiles_to_cache(vt, cfg, B)[:, :, :S]
    want = o.attention(0, qb.float().cpu().numpy().reshape(B, S, cfg.Hq, Dh), 0)
    tb.k_status_clear()
    tb.k_attn_select(3)
    try:
        tb.k_wait_test(2_000_000, 1)
        ob = torch.full((B * S, cfg.Hq * Dh), 768.0, dtype=torch.bfloat16, device=DEV)
        tb.k_attn(qb, kt, vt, ob, mc, B, S, 0, None)
        torch.cuda.synchronize()
        assert tb.k_attn_status() in (1, 2, 3)
        got = ob.float().cpu().numpy().reshape(B, S, cfg.Hq, Dh)
        untouched = got == 768.0
        # the grid's first CTA is the last query block (longest first) of head 0, sequence 0
        assert untouched[0, 128:, 0].all() and untouched.sum() == 128 * Dh
        done = ~untouched
        assert np.abs(got[done] - want[done]).max() < 2.0 ** -7 * np.abs(want).max() + 1e-6
    finally:
        tb.k_wait_test(0, -1)
        tb.k_status_clear()
    ob = torch.zeros((B * S, cfg.Hq * Dh), dtype=torch.bfloat16, device=DEV)
    tb.k_attn(qb, kt, vt, ob, mc, B, S, 0, None)
    torch.cuda.synchronize()
    tb.k_attn_select(0)
    assert tb.k_attn_status() == 0
    assert np.abs(ob.float().cpu().numpy().reshape(B, S, cfg.Hq, Dh) - want).max() < 2.0 ** -7 * np.abs(want).max() + 1e-6


def test_gemm_rejects_bad_arguments_and_accepts_empty():
    A = torch.zeros(8, 16, dtype=torch.bfloat16, device=DEV)
    Cd = torch.zeros(8, 8, dtype=torch.float32, device=DEV)
    with pytest.raises(tb.TgpError):
        tb.k_gemm(A, A, Cd, 8, 8, 12, 8, 0, 0)          # K % 8
    with pytest.raises(tb.TgpError):
        tb.k_gemm(A, A, Cd, 8, 8, 16, 8, 4, 0)          # col0 + n > ldc
    tb.k_gemm(A, A, Cd, 0, 8, 16, 8, 0, 0)              # empty M: no launch, no error
    torch.cuda.synchronize()


@pytest.mark.parametrize("M,d", [(1, 128), (5, 256), (37, 2048), (3, 8192)])
def test_rmsnorm_and_embed(M, d):
    V = 300
    tab_bits = rnd_bits(3, V * d).reshape(V, d)
    tok = (np.arange(M, dtype=np.int32) * 37 + 5) % V
    x = torch.empty(M, d, dtype=torch.float32, device=DEV)
    tb.k_embed(bf16_dev(tab_bits), torch.from_numpy(tok).to(DEV), x, M, d, V)
    torch.cuda.synchronize()
    assert np.array_equal(x.cpu().numpy(), si.bf16_bits_to_f32(tab_bits)[tok])
    assert tb.k_embed_status()[0] == 0
    xin = (np.random.default_rng(d).standard_normal((M, d)) * 3).astype(np.float32)
    g_bits = si.f32_to_bf16_bits(1.0 + 0.1 * np.random.default_rng(1).standard_normal(d).astype(np.float32))
    h = torch.empty(M, d, dtype=torch.bfloat16, device=DEV)
    tb.k_rmsnorm(torch.from_numpy(xin).to(DEV), d, bf16_dev(g_bits), h, M, d, 1e-5)
    torch.cuda.synchronize()
    o = oracle()
    want = o.rmsnorm(xin, si.bf16_bits_to_f32(g_bits).astype(np.float64))
    bf16_close(h.float().cpu().numpy(), want)


def test_embed_zeroes_rows_of_tokens_outside_the_vocabulary_and_records_the_first():
    """A token id outside [0, V) must never index the table (in an oversubscribed run the table may be mapped host
    memory): its row is zeros, the others are gathered as usual, and the error word names the row and the id."""
    V, d, M = 50, 64, 6
    tab_bits = rnd_bits(11, V * d).reshape(V, d)
    tok = np.array([3, V, 7, -1, 49, 2 ** 31 - 1], dtype=np.int32)
    x = torch.full((M, d), 7.0, dtype=torch.float32, device=DEV)
    tb.k_status_clear()
    tb.k_embed(bf16_dev(tab_bits), torch.from_numpy(tok).to(DEV), x, M, d, V)
    torch.cuda.synchronize()
    got = x.cpu().numpy()
    ok = (tok >= 0) & (tok < V)
    assert np.array_equal(got[ok], si.bf16_bits_to_f32(tab_bits)[tok[ok]])
    assert not got[~ok].any()
    bad, row, token = tb.k_embed_status()
    assert bad == 1 and row in (1, 3, 5) and token == int(tok[row])
    tb.k_status_clear()
    assert tb.k_embed_status()[0] == 0


def test_argmax_of_a_row_of_nans_is_a_legal_token():
    V = 5000
    lg = np.full((3, V), np.nan, dtype=np.float32)
    lg[1] = -np.inf
    lg[2, 4000] = 1.0
    am = torch.full((3,), -7, dtype=torch.int32, device=DEV)
    tb.k_argmax(torch.from_numpy(lg).to(DEV), am, 3, V)
    torch.cuda.synchronize()
    got = am.cpu().numpy()
    assert got[0] == 0 and got[1] == 0 and 0 <= got[2] < V


def make_tiles(cfg, B):
    nt = cfg.n_tiles
    k = [torch.zeros(B * cfg.Hkv * cfg.TK * cfg.Dh, dtype=torch.bfloat16, device=DEV) for _ in range(nt)]
    v = [torch.zeros(B * cfg.Hkv * cfg.TK * cfg.Dh, dtype=torch.bfloat16, device=DEV) for _ in range(nt)]
    return k, v


def tiles_to_cache(tiles, cfg, B):
    """[n_tiles] x [B, Hkv, TK, Dh] -> [B, Hkv, n_tiles*TK, Dh] fp32"""
    t = torch.stack([x.view(B, cfg.Hkv, cfg.TK, cfg.Dh) for x in tiles], dim=2)
    return t.reshape(B, cfg.Hkv, -1, cfg.Dh).float().cpu().numpy()


@pytest.mark.parametrize("attn_impl", [3, 2])
@pytest.mark.parametrize("Dh,Hq,Hkv,TK,S,T", [(64, 4, 2, 4, 9, 7), (128, 8, 2, 16, 40, 5), (64, 4, 4, 8, 33, 3), (128, 8, 1, 64, 130, 2),
                                             (64, 6, 2, 32, 70, 3)])      # three query heads per KV head: the per-head decode kernel
def test_rope_kv_and_attention_prefill_then_decode(Dh, Hq, Hkv, TK, S, T, attn_impl):
    B = 2
    tb.k_attn_select(attn_impl)
    cfg = replace(KCFG, Dh=Dh, Hq=Hq, Hkv=Hkv, TK=TK, S=S, T=T, B=B, d=Hq * Dh)
    lay_w = {(k, 0, -1): rnd_bits(k, 8).reshape(1, 8) for k in range(13)}
    o = OracleModel(cfg, lay_w)
    mc = model_cfg(cfg)
    cos = torch.empty(cfg.max_len * Dh // 2, dtype=torch.float32, device=DEV)
    sin = torch.empty_like(cos)
    tb.k_rope_tables(Dh, cfg.max_len, cfg.rope_base, cos, sin)
    assert np.array_equal(cos.cpu().numpy().reshape(cfg.max_len, Dh // 2), o.cos)
    kt, vt = make_tiles(cfg, B)
    scratch = torch.empty(tb.k_attn_scratch_bytes(mc) // 4, dtype=torch.float32, device=DEV)
    rng = np.random.default_rng(S)
    pos0 = 0
    for step in range(1 + T):
        q = S if step == 0 else 1
        q32 = rng.standard_normal((B * q, Hq * Dh)).astype(np.float32)
        k32 = rng.standard_normal((B * q, Hkv * Dh)).astype(np.float32)
        v32 = rng.standard_normal((B * q, Hkv * Dh)).astype(np.float32)
        qb = torch.empty(B * q, Hq * Dh, dtype=torch.bfloat16, device=DEV)
        ob = torch.empty(B * q, Hq * Dh, dtype=torch.bfloat16, device=DEV)
        tb.k_rope_kv(torch.from_numpy(q32).to(DEV), torch.from_numpy(k32).to(DEV), torch.from_numpy(v32).to(DEV), qb, kt, vt, cos, sin, mc, B, q, pos0)
        tb.k_attn(qb, kt, vt, ob, mc, B, q, pos0, scratch)
        torch.cuda.synchronize()
        # oracle: same steps
        qo = bf16_round(o.rope(q32.reshape(B, q, Hq, Dh), pos0))
        ko = bf16_round(o.rope(k32.reshape(B, q, Hkv, Dh), pos0))
        vo = bf16_round(v32.reshape(B, q, Hkv, Dh))
        o.K[0, :, :, pos0:pos0 + q] = ko.transpose(0, 2, 1, 3)
        o.V[0, :, :, pos0:pos0 + q] = vo.transpose(0, 2, 1, 3)
        bf16_close(qb.float().cpu().numpy().reshape(B, q, Hq, Dh), qo)
        got_k = tiles_to_cache(kt, cfg, B)[:, :, :pos0 + q]
        bf16_close(got_k, o.K[0, :, :, :pos0 + q])
        assert np.array_equal(tiles_to_cache(vt, cfg, B)[:, :, :pos0 + q], o.V[0, :, :, :pos0 + q].astype(np.float32))
        # attention on the oracle's own q and cache would differ by the rare rounding flips above; feed it the GPU's
        o.K[0, :, :, :pos0 + q] = got_k
        att = o.attention(0, qb.float().cpu().numpy().reshape(B, q, Hq, Dh), pos0)
        got = ob.float().cpu().numpy().reshape(B, q, Hq, Dh)
        assert np.abs(got - att).max() < 2.0 ** -7 * np.abs(att).max() + 1e-6
        assert np.mean(np.abs(got - bf16_round(att))) < 3e-3 * np.abs(att).mean()     # incl. the kernel's bf16 rounding of softmax weights
        pos0 += q
    tb.k_attn_select(0)


@pytest.mark.parametrize("Dh,Hq,Hkv,TK,S,B", [(64, 32, 8, 128, 512, 1), (128, 8, 2, 256, 300, 2), (64, 4, 4, 16, 100, 3)])
def test_tensor_core_prefill_attention_agrees_with_cuda_core_kernel(Dh, Hq, Hkv, TK, S, B):
    """Same q and KV tiles through all three prefill kernels.  The tensor-core kernels round the softmax weights to bf16
    before the second product (its one rounding the oracle does not mirror); outputs are bf16, so agreement is to a
    bf16 ulp, with a small mean difference."""
    cfg = replace(KCFG, Dh=Dh, Hq=Hq, Hkv=Hkv, TK=TK, S=S, T=0, B=B, d=Hq * Dh)
    mc = model_cfg(cfg)
    kt, vt = make_tiles(cfg, B)
    for j, (k, v) in enumerate(zip(kt, vt)):
        k.copy_(bf16_dev(rnd_bits(300 + j, k.numel())) * 30)
        v.copy_(bf16_dev(rnd_bits(400 + j, v.numel())) * 30)
    qb = (bf16_dev(rnd_bits(9, B * S * Hq * Dh)) * 30).view(B * S, Hq * Dh)
    outs = []
    for impl in (3, 2, 1):
        tb.k_attn_select(impl)
        ob = torch.zeros(B * S, Hq * Dh, dtype=torch.bfloat16, device=DEV)
        tb.k_attn(qb, kt, vt, ob, mc, B, S, 0, None)
        torch.cuda.synchronize()
        outs.append(ob.float().cpu().numpy())
    tb.k_attn_select(0)
    assert tb.k_attn_status() == 0
    ref = outs[2]
    assert np.abs(ref).max() > 0
    for a in outs[:2]:                                     # tcgen05 kernel, mma.sync kernel against the CUDA-core kernel
        assert np.isfinite(a).all()
        assert np.abs(a - ref).max() <= 2.0 ** -6 * np.abs(ref).max()
        assert np.abs(a - ref).mean() < 4e-3 * np.abs(ref).mean()


@pytest.mark.parametrize("Dh", [64, 128])
def test_tensor_core_prefill_attention_with_growing_scores(Dh):
    """Scores that grow along the sequence by far more than 2^8 per key block: the tcgen05 kernel has to move its
    exponent reference and rescale its TMEM accumulator at almost every block.  Checked against the oracle."""
    B, Hq, Hkv, TK, S = 2, 4, 2, 64, 400
    cfg = replace(KCFG, Dh=Dh, Hq=Hq, Hkv=Hkv, TK=TK, S=S, T=0, B=B, d=Hq * Dh)
    mc = model_cfg(cfg)
    o = OracleModel(cfg, {(k, 0, -1): rnd_bits(k, 8).reshape(1, 8) for k in range(13)})
    rng = np.random.default_rng(Dh)
    u = rng.standard_normal(Dh).astype(np.float32)
    u /= np.linalg.norm(u)
    ramp = (np.arange(S, dtype=np.float32) / 4.0)[None, None, :, None]                  # + ~16 in log2 units per 64 keys
    k32 = bf16_round(rng.standard_normal((B, Hkv, S, Dh)).astype(np.float32) + ramp * u)
    v32 = bf16_round(rng.standard_normal((B, Hkv, S, Dh)).astype(np.float32))
    q32 = bf16_round(rng.standard_normal((B, S, Hq, Dh)).astype(np.float32) + np.sqrt(Dh).astype(np.float32) * u)
    sgn = np.where(np.arange(Hq) % 2 == 0, 1.0, -1.0).astype(np.float32)[None, None, :, None]
    q32 = q32 * sgn                                                                     # odd heads: scores fall instead
    kt, vt = make_tiles(cfg, B)
    for t in range(cfg.n_tiles):
        lo, hi = t * TK, min(S, (t + 1) * TK)
        kt[t].view(B, Hkv, TK, Dh)[:, :, :hi - lo].copy_(torch.from_numpy(k32[:, :, lo:hi]).to(DEV))
        vt[t].view(B, Hkv, TK, Dh)[:, :, :hi - lo].copy_(torch.from_numpy(v32[:, :, lo:hi]).to(DEV))
    o.K[0, :, :, :S] = k32
    o.V[0, :, :, :S] = v32
    att = o.attention(0, q32, 0)
    qb = torch.from_numpy(q32.reshape(B * S, Hq * Dh)).to(DEV).bfloat16()
    for impl in (3, 2):
        tb.k_attn_select(impl)
        ob = torch.zeros(B * S, Hq * Dh, dtype=torch.bfloat16, device=DEV)
        tb.k_attn(qb, kt, vt, ob, mc, B, S, 0, None)
        torch.cuda.synchronize()
        got = ob.float().cpu().numpy().reshape(B, S, Hq, Dh)
        assert np.isfinite(got).all()
        assert np.abs(got - att).max() < 2.0 ** -6 * np.abs(att).max() + 1e-6
        assert np.mean(np.abs(got - bf16_round(att))) < 4e-3 * np.abs(att).mean()
    tb.k_attn_select(0)
    assert tb.k_attn_status() == 0


@pytest.mark.parametrize("Dh,TK", [(128, 64), (64, 128)])
def test_tensor_core_prefill_attention_of_a_later_chunk(Dh, TK):
    """A prompt processed in two chunks: the second chunk's queries start at position 192 and see the first chunk's keys
    unmasked plus their own causally.  Both tensor-core kernels against the oracle."""
    B, Hq, Hkv, P0, Q2 = 2, 4, 2, 192, 200
    S = P0 + Q2
    cfg = replace(KCFG, Dh=Dh, Hq=Hq, Hkv=Hkv, TK=TK, S=S, T=0, B=B, d=Hq * Dh)
    mc = model_cfg(cfg)
    o = OracleModel(cfg, {(k, 0, -1): rnd_bits(k, 8).reshape(1, 8) for k in range(13)})
    rng = np.random.default_rng(7 * Dh + TK)
    k32 = bf16_round(rng.standard_normal((B, Hkv, S, Dh)).astype(np.float32))
    v32 = bf16_round(rng.standard_normal((B, Hkv, S, Dh)).astype(np.float32))
    q32 = bf16_round(rng.standard_normal((B, Q2, Hq, Dh)).astype(np.float32))
    kt, vt = make_tiles(cfg, B)
    for t in range(cfg.n_tiles):
        lo, hi = t * TK, min(S, (t + 1) * TK)
        if lo < hi:
            kt[t].view(B, Hkv, TK, Dh)[:, :, :hi - lo].copy_(torch.from_numpy(k32[:, :, lo:hi]).to(DEV))
            vt[t].view(B, Hkv, TK, Dh)[:, :, :hi - lo].copy_(torch.from_numpy(v32[:, :, lo:hi]).to(DEV))
    o.K[0, :, :, :S] = k32
    o.V[0, :, :, :S] = v32
    att = o.attention(0, q32, P0)
    qb = torch.from_numpy(q32.reshape(B * Q2, Hq * Dh)).to(DEV).bfloat16()
    for impl in (3, 2):
        tb.k_attn_select(impl)
        ob = torch.zeros(B * Q2, Hq * Dh, dtype=torch.bfloat16, device=DEV)
        tb.k_attn(qb, kt, vt, ob, mc, B, Q2, P0, None)
        torch.cuda.synchronize()
        got = ob.float().cpu().numpy().reshape(B, Q2, Hq, Dh)
        assert np.abs(got - att).max() < 2.0 ** -7 * np.abs(att).max() + 1e-6
        assert np.mean(np.abs(got - bf16_round(att))) < 3e-3 * np.abs(att).mean()
    tb.k_attn_select(0)
    assert tb.k_attn_status() == 0


@pytest.mark.parametrize("Dh,Hq,Hkv,TK,kvlen,B", [(128, 32, 8, 256, 1280, 2), (128, 32, 8, 256, 1037, 3), (128, 64, 8, 64, 2112, 2), (64, 32, 8, 128, 640, 1),
                                                 (64, 4, 4, 16, 48, 1), (128, 8, 4, 32, 33, 2), (64, 8, 1, 16, 17, 4), (128, 4, 4, 48, 1, 2),
                                                 (64, 16, 2, 80, 401, 5)])
def test_tensor_core_decode_attention_matches_oracle_and_cuda_core_kernel(Dh, Hq, Hkv, TK, kvlen, B):
    """Decode attention on the tensor cores (forced wherever the geometry allows) against the oracle's softmax(q K^T) V on
    the same bf16 queries and cache, and against the CUDA-core kernel: contexts that end in the middle of a 16-key chunk,
    span many KV tiles and several CTAs per (sequence, KV head), groups of 1, 2, 4 and 8 query heads, a single key, and
    tiles whose bytes past the context are NaN (they must be neither read into the result nor multiplied by zero)."""
    cfg = replace(KCFG, Dh=Dh, Hq=Hq, Hkv=Hkv, TK=TK, S=kvlen, T=0, B=B, d=Hq * Dh)
    mc = model_cfg(cfg)
    kt, vt = make_tiles(cfg, B)
    assert len(kt) == (kvlen + TK - 1) // TK
    for j, (k, v) in enumerate(zip(kt, vt)):
        k.copy_(bf16_dev(rnd_bits(90 + j, k.numel())) * 40)
        v.copy_(bf16_dev(rnd_bits(190 + j, v.numel())) * 40)
    # everything past the context is poison
    last = kt[-1].view(B, Hkv, TK, Dh), vt[-1].view(B, Hkv, TK, Dh)
    used = kvlen - (len(kt) - 1) * TK
    if used < TK:
        last[0][:, :, used:, :] = float("nan")
        last[1][:, :, used:, :] = float("nan")
    qb = (bf16_dev(rnd_bits(7, B * Hq * Dh)) * 40).view(B, Hq * Dh)
    scratch = torch.empty(tb.k_attn_scratch_bytes(mc) // 4, dtype=torch.float32, device=DEV)
    outs = {}
    for impl in (2, 1):
        tb.k_attn_decode_select(impl)
        ob = torch.full((B, Hq * Dh), float("nan"), dtype=torch.bfloat16, device=DEV)
        tb.k_attn(qb, kt, vt, ob, mc, B, 1, kvlen - 1, scratch)
        torch.cuda.synchronize()
        outs[impl] = ob.float().cpu().numpy().reshape(B, 1, Hq, Dh)
    tb.k_attn_decode_select(0)
    o = OracleModel(cfg, {})
    kc, vc = tiles_to_cache(kt, cfg, B)[:, :, :kvlen], tiles_to_cache(vt, cfg, B)[:, :, :kvlen]
    o.K[0], o.V[0] = kc, vc
    att = o.attention(0, qb.float().cpu().numpy().reshape(B, 1, Hq, Dh), kvlen - 1)
    for impl, got in outs.items():
        assert np.isfinite(got).all(), impl
        assert np.abs(got - att).max() < 2.0 ** -7 * np.abs(att).max() + 1e-6, impl
        assert np.mean(np.abs(got - bf16_round(att))) < 3e-3 * np.abs(att).mean(), impl


# parts of a context in a cluster or through the scratch array: the last length that eight parts take and the first that more do, few KV tiles (one
# and two, which the scratch array would limit; five), numbers of parts that are not a power of two, eight query heads per KV head
@pytest.mark.parametrize("Dh,Hq,Hkv,TK,kvlen,B,launches", [(64, 4, 4, 64, 3072, 1, 1), (64, 4, 4, 64, 3073, 1, 2), (128, 8, 1, 1024, 5000, 1, 1), (128, 32, 8, 256, 4000, 4, 2),
                                                           (64, 8, 8, 64, 330, 2, 1), (128, 64, 8, 64, 900, 4, 1), (128, 16, 8, 64, 3100, 2, 2), (128, 8, 8, 64, 1500, 8, 1),
                                                           (128, 32, 8, 2048, 4000, 4, 1), (64, 40, 40, 4096, 1100, 2, 1), (128, 32, 8, 800, 4000, 4, 2)])
def test_parts_of_a_decode_context_in_clusters_and_in_the_scratch_array(Dh, Hq, Hkv, TK, kvlen, B, launches):
    cfg = replace(KCFG, Dh=Dh, Hq=Hq, Hkv=Hkv, TK=TK, S=kvlen, T=0, B=B, d=Hq * Dh)
    gen = torch.Generator(device=DEV)
    gen.manual_seed(kvlen + B)
    n = (kvlen + TK - 1) // TK
    kt, vt = ([torch.randn((B * Hkv * TK, Dh), device=DEV, generator=gen).bfloat16() for _ in range(n)] for _ in range(2))
    q = torch.randn((B, Hq * Dh), device=DEV, generator=gen).bfloat16()
    scratch = torch.full((tb.k_attn_scratch_bytes(model_cfg(cfg)) // 4,), 7.0, device=DEV)
    ob = torch.full((B, Hq * Dh), float("nan"), dtype=torch.bfloat16, device=DEV)
    tb.k_attn(q, kt, vt, ob, model_cfg(cfg), B, 1, kvlen - 1, scratch)
    torch.cuda.synchronize()
    assert bool((scratch == 7.0).all()) == (launches == 1)         # parts of a cluster do not touch it
    K, V = (torch.stack([t.view(B, Hkv, TK, Dh) for t in ts], dim=2).reshape(B, Hkv, n * TK, Dh)[:, :, :kvlen].double().repeat_interleave(Hq // Hkv, dim=1) for ts in (kt, vt))
    want = (torch.softmax(q.double().view(B, Hq, 1, Dh) @ K.transpose(-1, -2) / Dh ** 0.5, -1) @ V).reshape(B, Hq * Dh)
    # half a bf16 step of the output and of each of the probabilities, whose roundings average out: 2^-9 of the largest V, as in the tests above
    assert float((ob.double() - want).abs().max()) < 2.0 ** -7 * float(want.abs().max()) + 1e-6
    assert float((ob.double() - want).abs().mean()) < 5e-3 * float(want.abs().mean())


def test_attention_single_key_returns_v():
    cfg = replace(KCFG, B=1, S=1, T=0)
    mc = model_cfg(cfg)
    kt, vt = make_tiles(cfg, 1)
    vt[0].copy_(bf16_dev(rnd_bits(9, vt[0].numel())))
    kt[0].copy_(bf16_dev(rnd_bits(8, kt[0].numel())))
    qb = bf16_dev(rnd_bits(7, cfg.Hq * cfg.Dh)).view(1, -1)
    for scratch in (None, torch.empty(tb.k_attn_scratch_bytes(mc) // 4, dtype=torch.float32, device=DEV)):
        ob = torch.empty(1, cfg.Hq * cfg.Dh, dtype=torch.bfloat16, device=DEV)
        tb.k_attn(qb, kt, vt, ob, mc, 1, 1, 0, scratch)
        torch.cuda.synchronize()
        v = vt[0].view(1, cfg.Hkv, cfg.TK, cfg.Dh)[0, :, 0]                     # first token of each kv head
        want = v.repeat_interleave(cfg.Hq // cfg.Hkv, dim=0).reshape(1, -1)
        assert torch.equal(ob, want)


def test_swiglu_and_argmax():
    n = 4 * 1000 + 4
    rng = np.random.default_rng(4)
    g = (rng.standard_normal(n) * 4).astype(np.float32)
    u = rng.standard_normal(n).astype(np.float32)
    out = torch.empty(n, dtype=torch.bfloat16, device=DEV)
    tb.k_swiglu(torch.from_numpy(g).to(DEV), torch.from_numpy(u).to(DEV), out, n)
    torch.cuda.synchronize()
    gd = g.astype(np.float64)
    bf16_close(out.float().cpu().numpy(), bf16_round((gd / (1 + np.exp(-gd)) * u).astype(np.float32)))
    B, V = 5, 128256
    lg = rng.standard_normal((B, V)).astype(np.float32)
    lg[1, 77] = lg[1, 90000] = 9.0            # tie: lowest index wins
    lg[2, :] = 0.5                            # all equal -> 0
    lg[3, V - 1] = 11.0                       # last element
    am = torch.empty(B, dtype=torch.int32, device=DEV)
    tb.k_argmax(torch.from_numpy(lg).to(DEV), am, B, V)
    torch.cuda.synchronize()
    assert am.cpu().numpy().tolist() == np.argmax(lg, axis=1).tolist()
    assert am.cpu().numpy()[1] == 77 and am.cpu().numpy()[2] == 0 and am.cpu().numpy()[3] == V - 1


def test_overlapping_gemv_launches_keep_their_dependencies():
    """Back-to-back weight-streaming launches accumulate into the same output (each depends on the one before through C).
    With dependent-launch overlap a launch starts loading weights early but must not touch C before its predecessor has
    finished: the chain must give bit-identical results with overlap on and off, and equal the oracle's sum."""
    M, n, K, reps = 2, 4100, 2048, 12
    a_bits = rnd_bits(21, M * K).reshape(M, K)
    A = bf16_dev(a_bits)
    Ws = [rnd_bits(30 + i, n * K).reshape(n, K) for i in range(3)]
    Wd = [bf16_dev(w) for w in Ws]
    outs = []
    for overlap in (1, 0):
        tb.k_gemv_overlap(overlap)
        Cd = torch.zeros(M, n, dtype=torch.float32, device=DEV)
        for i in range(reps):
            tb.k_gemm(A, Wd[i % 3], Cd, M, n, K, n, 0, 1)
        torch.cuda.synchronize()
        outs.append(Cd.cpu().numpy())
    tb.k_gemv_overlap(1)
    assert np.array_equal(outs[0], outs[1])
    o = oracle()
    a = si.bf16_bits_to_f32(a_bits)
    want = sum(o.linear(a, si.bf16_bits_to_f32(Ws[i % 3]).astype(np.float64)).astype(np.float64) for i in range(reps))
    assert np.abs(outs[0] - want).max() < 1e-4 * np.abs(want).max()


def test_chained_products_read_their_activations_early_with_the_same_bits():
    """Under the caller's promise (tgp_k_gemm_chain) a product that directly follows another one over the same activations
    requests them before its predecessor has finished.  The chain must give the bits of unchained launches; a product
    that follows a kernel which rewrote the activations (an RMSNorm of this library) is not chained and sees the new values."""
    M, n, K = 8, 1152, 4096
    rng = np.random.default_rng(77)
    x0 = torch.from_numpy(rng.standard_normal((M, K)).astype(np.float32)).to(DEV)
    gain = bf16_dev(rnd_bits(78, K))
    A = torch.empty(M, K, dtype=torch.bfloat16, device=DEV)
    Ws = [bf16_dev(rnd_bits(80 + i, n * K).reshape(n, K)) for i in range(4)]
    outs = []
    for chain in (0, 1):
        tb.k_gemm_chain(chain)
        x = x0.clone()
        res = []
        for rep in range(3):
            tb.k_rmsnorm(x, K, gain, A, M, K, 1e-5)               # rewrites A: the product after it waits for it
            x.mul_(1.25)                                          # (another stream op between the repetitions; before the norm, not between products)
            Cs = [torch.zeros(M, n, dtype=torch.float32, device=DEV) for _ in Ws]
            for W, C in zip(Ws, Cs):
                tb.k_gemm(A, W, C, M, n, K, n, 0, 0)
            torch.cuda.synchronize()
            res.append([c.cpu().numpy() for c in Cs])
        outs.append(res)
    tb.k_gemm_chain(0)
    for rep in range(3):
        for a, b in zip(outs[0][rep], outs[1][rep]):
            assert np.array_equal(a, b)
    assert not np.array_equal(outs[0][0][0], outs[0][1][0])          # the activations did change between repetitions


@pytest.mark.parametrize("M,ns,K,grouped", [
    (1, (2048, 512, 512), 2048, True),            # the q, k, v projections of the 1B shape: one launch
    (2, (300, 7, 129, 1), 264, True),             # four ragged parts, K not a multiple of the chunk
    (1, (4096, 8192), 4096, False),               # a block of many rows is launched alone
    (2, (640, 640, 64), 8192, False),             # long K at M <= 2: the parts take the split-K kernel, alone
    (8, (1152, 1152, 1152, 640), 14336, True),    # the pieces of an 8B down projection: 8-row CTAs, 16 warps
    (16, (512,) * 8, 28672, True),                # eight pieces of a 70B down projection
    (8, (1024, 1024), 4096, True),                # k and v of the 8B shape
    (8, (4096, 1024, 1024), 4096, True),          # q, k and v of the 8B shape: all take the persistent 16-warp kernel
    (8, (4096, 4096, 4096, 2048, 4096, 4096, 4096, 2048), 4096, True),   # gate and up of the 8B shape in 32 MiB pieces
    (8, (8192, 1024), 2048, False),               # a piece of many rows takes the 8-warp kernel: one launch each
    (32, (500, 260, 33), 160, True),              # ragged row counts, four groups of activation rows
    (5, (24000, 64), 64, False),                  # a block that fills the machine alone
    (40, (256, 256), 512, False)])                # more activation rows than the skinny kernels take
@pytest.mark.parametrize("accumulate", [0, 1])
def test_grouped_products_equal_single_products_and_oracle(M, ns, K, grouped, accumulate):
    """Products that share their activations: the grouped call must give the bits of one tgp_k_gemm() call per part,
    whether it runs as one launch or falls back to one launch per part, with the switch on and off, and leave the
    columns beyond each part untouched; the values are checked against the oracle's linear()."""
    keys = {tb.k_gemm_group_key(M, n, K) for n in ns}
    assert (len(keys) == 1 and 0 not in keys) == grouped
    a_bits = rnd_bits(51, M * K).reshape(M, K)
    A = bf16_dev(a_bits)
    w_bits = [rnd_bits(60 + s, n * K).reshape(n, K) for s, n in enumerate(ns)]
    Wd = [bf16_dev(w) for w in w_bits]
    ldcs = [n + 8 * (s + 1) for s, n in enumerate(ns)]
    c0 = [np.random.default_rng(100 + s).standard_normal((M, ld)).astype(np.float32) * 0.01 for s, ld in enumerate(ldcs)]
    fresh = lambda: [torch.from_numpy(c.copy()).to(DEV) for c in c0]
    single = fresh()
    for s, n in enumerate(ns):
        tb.k_gemm(A, Wd[s], single[s], M, n, K, ldcs[s], 0, accumulate)
    outs = []
    for enable in (1, 0):
        tb.k_gemm_group_select(enable)
        out = fresh()
        tb.k_gemm_group(A, Wd, out, M, list(ns), K, ldcs, accumulate)
        torch.cuda.synchronize()
        outs.append([g.cpu().numpy() for g in out])
        assert enable or tb.k_gemm_group_key(M, ns[0], K) == 0
    tb.k_gemm_group_select(1)
    o = oracle()
    a = si.bf16_bits_to_f32(a_bits)
    for s, n in enumerate(ns):
        ref = single[s].cpu().numpy()
        assert np.array_equal(outs[0][s], ref) and np.array_equal(outs[1][s], ref)
        assert np.array_equal(ref[:, n:], c0[s][:, n:])
        want = o.linear(a, si.bf16_bits_to_f32(w_bits[s]).astype(np.float64)).astype(np.float64) + (c0[s][:, :n] if accumulate else 0)
        assert np.abs(ref[:, :n] - want).max() < 2e-5 * max(np.abs(want).max(), 0.01) + 1e-7
    if M == 1 and accumulate == 0:
        with pytest.raises(tb.TgpError):
            tb.k_gemm_group(A, Wd[:1] * 9, [single[0]] * 9, M, [ns[0]] * 9, K, [ldcs[0]] * 9)      # more parts than the call takes
        with pytest.raises(tb.TgpError):
            tb.k_gemm_group(A, Wd[:2], single[:2], M, [ns[0], ns[1]], K, [ns[0] - 1, ldcs[1]])       # row stride below the part's width


@pytest.mark.parametrize("M,n,K", [(3, 100, 64), (8, 4096, 4096), (8, 1030, 512), (13, 77, 128), (16, 260, 1024), (17, 64, 96), (24, 2049, 2048),
                                   (32, 4100, 8192), (5, 16, 32),
                                   # few rows and long K: the split-K kernel (K divided among the warps of a CTA; ragged rows, K that
                                   # leaves the last warps without a chunk)
                                   (8, 1152, 14336), (5, 650, 14368), (16, 1024, 4096), (9, 24, 2080), (8, 16, 16384)])
@pytest.mark.parametrize("accumulate", [0, 1])
def test_skinny_tensor_core_gemv_matches_oracle_and_cuda_core_path(M, n, K, accumulate):
    a_bits, w_bits = rnd_bits(41, M * K).reshape(M, K), rnd_bits(42, n * K).reshape(n, K)
    A, W = bf16_dev(a_bits), bf16_dev(w_bits)
    c0 = np.random.default_rng(M + n).standard_normal((M, n + 8)).astype(np.float32) * 0.01
    outs, names = [], []
    for impl in (0, 1):
        (tb.k_skinny_select if M <= 16 else tb.k_gemm_select)(impl)          # (17 rows and more are the tcgen05 kernels', 1: the CUDA-core tiles)
        Cd = torch.from_numpy(c0.copy()).to(DEV)
        tb.k_gemm(A, W, Cd, M, n, K, n + 8, 4, accumulate)
        torch.cuda.synchronize()
        outs.append(Cd.cpu().numpy())
        names.append(tb.k_gemm_last_kernel())
    tb.k_skinny_select(0)
    tb.k_gemm_select(0)
    assert names[0] != names[1]
    want = c0.astype(np.float64).copy()
    prod = oracle().linear(si.bf16_bits_to_f32(a_bits), si.bf16_bits_to_f32(w_bits).astype(np.float64)).astype(np.float64)
    want[:, 4:4 + n] = prod + (c0[:, 4:4 + n] if accumulate else 0)
    scale = max(np.abs(prod).max(), 0.01)
    assert np.abs(outs[0] - want).max() < 2e-5 * scale + 1e-7
    assert np.abs(outs[0] - outs[1]).max() < 2e-5 * scale + 1e-7
    for out in outs:
        assert np.array_equal(out[:, :4], c0[:, :4]) and np.array_equal(out[:, 4 + n:], c0[:, 4 + n:])


# blocks on either side of the lines that send a product of 3 - 16 rows to the persistent list kernel: K below / at 2048 and 3072
# (M <= 8) and 4096 (M <= 16), row counts around five 16-row groups per SM, a ragged last group, a K that ends inside a warp's chunk
@pytest.mark.parametrize("M,ns,K,listed_family", [(3, (4737,), 3072, 1), (8, (4800, 4737), 3104, 1), (8, (11840, 12000), 2048, 1), (5, (11800,), 2080, 0), (9, (4737, 5000), 4096, 1),
                                                  (16, (4737, 8064), 4128, 1), (13, (8064,), 4096, 1), (12, (4737, 8064), 4064, 0)])
def test_blocks_of_many_rows_take_the_list_kernel_with_the_same_bits_alone_and_in_a_list(M, ns, K, listed_family):
    assert all(tb.k_gemm_group_key(M, n, K) >> 24 == listed_family for n in ns)      # 1: the list kernel, 0: alone in another one
    gen = torch.Generator(device=DEV)
    gen.manual_seed(M * K + len(ns))
    A = torch.randn((M, K), device=DEV, generator=gen).bfloat16()
    Ws = [(torch.randn((n, K), device=DEV, generator=gen) * 0.02).bfloat16() for n in ns]
    c0 = [torch.randn((M, n), device=DEV, generator=gen) for n in ns]
    alone, listed = [c.clone() for c in c0], [c.clone() for c in c0]
    for W, C, n in zip(Ws, alone, ns):
        tb.k_gemm(A, W, C, M, n, K, n, 0, True)
    tb.k_gemm_group(A, Ws, listed, M, list(ns), K, list(ns), True)
    torch.cuda.synchronize()
    for W, a, b, c in zip(Ws, alone, listed, c0):
        assert torch.equal(a, b)
        want = A.double() @ W.double().T + c.double()
        # fp32 sums of K products of N(0, 1) x N(0, 0.02): errors of a few 2^-24 of the partial sums' size, bounded as in the tests above
        assert float((a.double() - want).abs().max()) < 2e-5 * float(want.abs().max())


# two row groups per CTA (4096 and 2 x 2048 rows on 148 SMs: 128 CTAs of 32 rows) and one
@pytest.mark.parametrize("M,ns,K", [(16, (4096,), 4096), (9, (2048, 2048), 1024), (16, (1024, 1000), 1024)])
def test_products_of_9_to_16_rows_take_no_more_shared_memory_than_their_partial_tiles(M, ns, K, tmp_path):
    A = torch.ones((M, K), device=DEV, dtype=torch.bfloat16)
    Ws, Cs = [torch.ones((n, K), device=DEV, dtype=torch.bfloat16) for n in ns], [torch.empty((M, n), device=DEV) for n in ns]
    launched = kernels_of(lambda: tb.k_gemm_group(A, Ws, Cs, M, list(ns), K, list(ns)), tmp_path)
    assert len(launched) == 1 and "tgp_wstream_mma_group_kernel" in launched[0][0]
    assert launched[0][1]["shared memory"] in (16 << 10, 32 << 10)          # 16 warps x 1 or 2 groups x 16 x 16 sums, which a kernel may declare


# one and two rows on blocks of many rows, on either side of what is listed (K of two to four times 2048 columns at one row, up to 8704 weight rows and K a multiple of 2048 at two)
@pytest.mark.parametrize("M,ns,K,listed", [(1, (4736, 5001), 4096, True), (1, (9000, 4737), 8192, True), (1, (4800, 4736), 6144, True), (1, (5000, 4736), 4104, False),
                                           (1, (5000, 4736), 10240, False), (2, (8704, 4736, 8192), 2048, True), (2, (4740, 8705), 2048, False), (2, (8704, 4736), 520, False),
                                           (2, (4736, 4736), 8192, True)])
@pytest.mark.parametrize("accumulate", [False, True])
def test_blocks_of_many_rows_at_one_and_two_activation_rows(M, ns, K, listed, accumulate):
    keys = {tb.k_gemm_group_key(M, n, K) for n in ns}
    assert (len(keys) == 1 and 0 not in keys) == listed
    gen = torch.Generator(device=DEV)
    gen.manual_seed(M * K + len(ns))
    A = torch.randn((M, K), device=DEV, generator=gen).bfloat16()
    Ws = [(torch.randn((n, K), device=DEV, generator=gen) * 0.02).bfloat16() for n in ns]
    c0 = [torch.randn((M, n + 4), device=DEV, generator=gen) for n in ns]
    alone, listed_c = [c.clone() for c in c0], [c.clone() for c in c0]
    for W, C, n in zip(Ws, alone, ns):
        tb.k_gemm(A, W, C, M, n, K, n + 4, 0, accumulate)
    tb.k_gemm_group(A, Ws, listed_c, M, list(ns), K, [n + 4 for n in ns], accumulate)
    torch.cuda.synchronize()
    for W, a, b, c, n in zip(Ws, alone, listed_c, c0, ns):
        assert torch.equal(a, b) and torch.equal(a[:, n:], c[:, n:])
        want = A.double() @ W.double().T + (c[:, :n].double() if accumulate else 0)
        # lane-strided fp32 sums of K products: a few 2^-24 of the partial sums' size, as in the tests below
        assert float((a[:, :n].double() - want).abs().max()) < 2e-5 * float(want.abs().max())


# on 148 SMs, one wave being 7104 rows: up to three quarters of one, and the beginning of the second
@pytest.mark.parametrize("n,K,listed", [(4736, 2048, True), (5328, 4096, True), (5329, 4096, False), (7104, 2048, False), (7105, 2048, True), (8704, 6144, True),
                                        (8705, 6144, False), (5328, 3072, False)])
def test_two_activation_rows_share_a_launch_where_the_last_wave_is_emptier(n, K, listed, tmp_path):
    assert (tb.k_gemm_group_key(2, n, K) != 0) == listed
    gen = torch.Generator(device=DEV)
    gen.manual_seed(n + K)
    A = torch.randn((2, K), device=DEV, generator=gen).bfloat16()
    Ws = [(torch.randn((n, K), device=DEV, generator=gen) * 0.02).bfloat16() for _ in range(2)]
    alone, together = ([torch.empty((2, n), device=DEV) for _ in Ws] for _ in range(2))
    for W, C in zip(Ws, alone):
        tb.k_gemm(A, W, C, 2, n, K, n, 0, False)
    launched = kernels_of(lambda: tb.k_gemm_group(A, Ws, together, 2, [n, n], K, [n, n]), tmp_path)
    assert [("group" in name) for name, _ in launched] == ([True] if listed else [False, False])
    assert all(torch.equal(a, b) for a, b in zip(alone, together))


# on 148 SMs: waves of 3552 rows (a row per warp) and 9472 (two), the fuller last wave
@pytest.mark.parametrize("n,K,rows_per_warp", [(7104, 4096, 1), (7105, 8192, 2), (9472, 6144, 2), (9473, 6144, 1), (8192, 2048, 2), (10240, 10240, 2)])
def test_one_activation_row_takes_the_kernel_whose_last_wave_is_fuller_with_the_same_bits(n, K, rows_per_warp, tmp_path):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(n + K)
    A = torch.randn((1, K), device=DEV, generator=gen).bfloat16()
    W = (torch.randn((n, K), device=DEV, generator=gen) * 0.02).bfloat16()
    alone, parts = torch.empty((1, n), device=DEV), torch.empty((1, n), device=DEV)
    (name, _), = kernels_of(lambda: tb.k_gemm(A, W, alone, 1, n, K, n, 0, False), tmp_path)
    assert f"tgp_wstream_kernel<1, {rows_per_warp}, " in name
    at = [0, 4000, n]                                      # pieces of fewer than 4736 rows: a row per warp, or K split over warps
    for lo, hi in zip(at, at[1:]):
        tb.k_gemm(A, W[lo:hi], parts, 1, hi - lo, K, n, lo, False)
    want = A.double() @ W.double().T
    for got in (alone, parts):
        # lane-strided fp32 sums of K products: a few 2^-24 of the partial sums' size, as in the tests above
        assert float((got.double() - want).abs().max()) < 2e-5 * float(want.abs().max())
    assert K >= 8192 or torch.equal(alone[:, :4000], parts[:, :4000])


# the list kernel at 9 - 16 rows around a chunk of 16 warps x 128 columns (one column block, a warp's chunk more or less, many chunks), ragged
# row groups, one and two row groups per CTA; and lists of which only neighbours share a kernel
@pytest.mark.parametrize("M,ns,K", [(9, (1, 17), 32), (16, (1024, 1000), 1024), (12, (300,), 2016), (16, (2048, 4100), 2048), (11, (33, 640), 2080), (16, (500,), 14368),
                                    (16, (8200, 1024, 1000), 4096), (10, (1000, 4800, 4736, 7), 2048), (9, (16, 8065, 8070, 16, 24), 4096)])
@pytest.mark.parametrize("accumulate", [False, True])
def test_products_of_9_to_16_rows_alone_and_in_lists_of_several_kernels(M, ns, K, accumulate):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(M * K + len(ns))
    A = torch.randn((M, K), device=DEV, generator=gen).bfloat16()
    Ws = [(torch.randn((n, K), device=DEV, generator=gen) * 0.02).bfloat16() for n in ns]
    lds = [n + 4 * (s % 3) for s, n in enumerate(ns)]
    c0 = [torch.randn((M, ld), device=DEV, generator=gen) for ld in lds]
    alone, listed = [c.clone() for c in c0], [c.clone() for c in c0]
    for W, C, n, ld in zip(Ws, alone, ns, lds):
        tb.k_gemm(A, W, C, M, n, K, ld, 0, accumulate)
    tb.k_gemm_group(A, Ws, listed, M, list(ns), K, lds, accumulate)
    torch.cuda.synchronize()
    for W, a, b, c, n in zip(Ws, alone, listed, c0, ns):
        assert torch.equal(a, b) and torch.equal(a[:, n:], c[:, n:])
        want = A.double() @ W.double().T + (c[:, :n].double() if accumulate else 0)
        # fp32 sums of K products of N(0, 1) x N(0, 0.02): errors of a few 2^-24 of the partial sums' size, bounded as in the tests above
        assert float((a[:, :n].double() - want).abs().max()) < 2e-5 * float(want.abs().max()) + 1e-7


# which neighbours of a list share a launch: those of one key, whatever stands between others (q of a wide model takes the tcgen05 kernel at 16
# rows, its k and v the list kernel); at most eight blocks
@pytest.mark.parametrize("M,ns,K,kernels", [(16, (8200, 1024, 1000), 4096, ["wstream_tc", "mma_group"]), (9, (16, 8065, 8070, 16, 24), 4096, ["mma_group", "wstream_tc", "mma_group"]),
                                            (12, (1000, 8200, 1000), 4096, ["mma_group", "wstream_tc", "mma_group"]), (10, (64,) * 8, 2048, ["mma_group"]),
                                            (1, (4736, 5000), 4096, ["wstream_group"]), (1, (4736, 64, 4736), 4096, ["wstream_kernel", "wstream_kernel", "wstream_kernel"]),
                                            (2, (64, 100, 4736, 4736), 4096, ["wstream_group", "wstream_group"]), (1, (5000, 4736), 10240, ["wstream_kernel", "wstream_kernel"]),
                                            (200, (256, 256), 1024, ["tc"])])
def test_neighbours_of_one_key_share_a_launch(M, ns, K, kernels, tmp_path):
    A = torch.ones((M, K), device=DEV, dtype=torch.bfloat16)
    Ws, Cs = [torch.ones((n, K), device=DEV, dtype=torch.bfloat16) for n in ns], [torch.zeros((M, n), device=DEV) for n in ns]
    call = lambda: tb.k_gemm_group(A, Ws, Cs, M, list(ns), K, list(ns))
    launched = [name for name, _ in kernels_of(call, tmp_path)]
    assert len(launched) == len(kernels) and all(k in name for k, name in zip(kernels, launched)), launched
    assert all(bool((C == K).all()) for C in Cs)
    tb.k_gemm_group_select(0)
    try:
        assert len(kernels_of(call, tmp_path)) == len(ns)
    finally:
        tb.k_gemm_group_select(1)


# the tcgen05 kernels on either side of their dispatch lines: one tile per CTA unsplit / in 2 / in 4 slices of K (ragged row tiles, K that
# ends inside a 64-wide block or leaves slices of unequal length), the line at 8192 columns above 128 activation rows, the paired
# kernel's activation tiles (one of 160 rows, three of 224, the last one ragged), lists of ragged parts
@pytest.mark.parametrize("M,ns,K", [(17, (4736, 129), 1024), (33, (130, 1), 1032), (61, (9400, 4737), 1024), (64, (9473,), 2048), (128, (4737,), 8192),
                                    (16, (8065, 8193), 512), (129, (257, 255), 8184), (129, (257, 255), 8192), (300, (2300,), 8200), (603, (300, 513), 1096),
                                    (100, (33,) * 8, 1024)])
@pytest.mark.parametrize("accumulate", [False, True])
def test_tcgen05_products_alone_and_in_a_list(M, ns, K, accumulate):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(M * K + len(ns))
    A = torch.randn((M, K), device=DEV, generator=gen).bfloat16()
    Ws = [(torch.randn((n, K), device=DEV, generator=gen) * 0.02).bfloat16() for n in ns]
    lds = [n + 4 * (s % 3) for s, n in enumerate(ns)]
    c0 = [torch.randn((M, ld), device=DEV, generator=gen) for ld in lds]
    alone, listed = [c.clone() for c in c0], [c.clone() for c in c0]
    for W, C, n, ld in zip(Ws, alone, ns, lds):
        tb.k_gemm(A, W, C, M, n, K, ld, 0, accumulate)
    tb.k_gemm_group(A, Ws, listed, M, list(ns), K, lds, accumulate)
    torch.cuda.synchronize()
    assert tb.k_gemm_status() == 0
    for W, a, b, c, n in zip(Ws, alone, listed, c0, ns):
        assert torch.equal(a, b) and torch.equal(a[:, n:], c[:, n:])
        want = A.double() @ W.double().T + (c[:, :n].double() if accumulate else 0)
        assert float((a[:, :n].double() - want).abs().max()) < 2e-5 * float(want.abs().max())


def test_tcgen05_product_in_slices_gives_up_on_a_wait_that_runs_out_and_recovers():
    """The one-tile-per-CTA kernel with K in four slices: the grid's first CTA never loads its second block, so the waits for its
    tile run out; no CTA of its cluster stores anything, every other tile is right, and the next launch is correct."""
    M, n, K = 61, 300, 2048
    A, W = bf16_dev(rnd_bits(53, M * K).reshape(M, K)), bf16_dev(rnd_bits(54, n * K).reshape(n, K))
    want = (A.double() @ W.double().T).cpu().numpy()
    SENT = 12345.0
    tb.k_status_clear()
    try:
        tb.k_wait_test(2_000_000, 1)
        Cd = torch.full((M, n), SENT, dtype=torch.float32, device=DEV)
        tb.k_gemm(A, W, Cd, M, n, K, n, 0, 0)
        torch.cuda.synchronize()
        assert tb.k_gemm_status() != 0
        got = Cd.cpu().numpy()
        assert (got[:, :128] == SENT).all()
        assert np.abs(got[:, 128:] - want[:, 128:]).max() < 2e-5 * np.abs(want).max()
    finally:
        tb.k_wait_test(0, -1)
        tb.k_status_clear()
    Cd = torch.zeros((M, n), dtype=torch.float32, device=DEV)
    tb.k_gemm(A, W, Cd, M, n, K, n, 0, 0)
    torch.cuda.synchronize()
    assert tb.k_gemm_status() == 0
    assert np.abs(Cd.cpu().numpy() - want).max() < 2e-5 * np.abs(want).max()


@pytest.mark.parametrize("d", [1024, 1028, 2048, 2052, 4096, 4100, 8192, 8196])
@pytest.mark.parametrize("M,shift", [(3, 0), (2, 2), (2049, 0)])
def test_rmsnorm_row_lengths_around_its_register_variants(d, M, shift):
    """Row lengths at and just past what the variants hold in registers, a row stride longer than the row, gains and outputs
    that are 4-byte but not 8-byte aligned (shift), many long rows."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(d + M)
    x = torch.randn((M, d + 4), device=DEV, generator=gen) * 3
    g = (1 + 0.1 * torch.randn(d + shift, device=DEV, generator=gen)).bfloat16()[shift:]
    h = torch.zeros(M * d + shift, dtype=torch.bfloat16, device=DEV)
    tb.k_rmsnorm(x, d + 4, g, h[shift:], M, d, 1e-5)
    torch.cuda.synchronize()
    xd = x[:, :d].double()
    want = xd / torch.sqrt((xd * xd).mean(dim=1, keepdim=True) + 1e-5) * g.double()
    bf16_close(h[shift:].view(M, d).float().cpu().numpy(), want.float().bfloat16().float().cpu().numpy())


@pytest.mark.parametrize("Dh,shift", [(64, 0), (128, 0), (128, 2), (32, 0)])
@pytest.mark.parametrize("B,S,pos0", [(1, 1, 0), (3, 1, 70), (2, 37, 50), (1, 700, 3)])
def test_rope_and_kv_append_vector_and_general_forms(Dh, shift, B, S, pos0):
    """The four-dimensions-a-thread form and the general one (a head size it does not serve, a query buffer that is not 16-byte
    aligned) against double precision: positions across tile edges, one CTA and several per position."""
    Hq, Hkv, TK = 6, 2, 16
    cfg = replace(KCFG, Dh=Dh, Hq=Hq, Hkv=Hkv, TK=TK, S=S, T=0, B=B, d=Hq * Dh)
    cfg = replace(cfg, S=S + pos0)
    mc = model_cfg(cfg)
    nt = (pos0 + S + TK - 1) // TK
    gen = torch.Generator(device=DEV)
    gen.manual_seed(Dh + S)
    q, k, v = (torch.randn((B * S, h * Dh), device=DEV, generator=gen) for h in (Hq, Hkv, Hkv))
    kt, vt = ([torch.full((B * Hkv * TK, Dh), 5.0, dtype=torch.bfloat16, device=DEV) for _ in range(nt)] for _ in range(2))
    cos, sin = (torch.randn((pos0 + S, Dh // 2), device=DEV, generator=gen) for _ in range(2))
    qb = torch.zeros(B * S * Hq * Dh + shift, dtype=torch.bfloat16, device=DEV)
    tb.k_rope_kv(q, k, v, qb[shift:], kt, vt, cos, sin, mc, B, S, pos0)
    torch.cuda.synchronize()

    def rot(x, h):
        x = x.double().view(B, S, h, Dh)
        c, s_ = cos[pos0:].double().view(1, S, 1, -1), sin[pos0:].double().view(1, S, 1, -1)
        a, b = x[..., :Dh // 2], x[..., Dh // 2:]
        return torch.cat([a * c - b * s_, b * c + a * s_], dim=-1)

    # half a bf16 step of the result, plus the fp32 rounding of two products of factors below 6 (3 x 36 x 2^-24), which is what is
    # left where they cancel
    close = lambda got, want: bool(((got.double() - want).abs() <= 2.0 ** -8 * want.abs() + 1e-5).all())
    assert close(qb[shift:].view(B, S, Hq, Dh), rot(q, Hq))
    for tiles, want in ((kt, rot(k, Hkv)), (vt, v.double().view(B, S, Hkv, Dh))):
        cache = torch.stack([t.view(B, Hkv, TK, Dh) for t in tiles], dim=2).reshape(B, Hkv, nt * TK, Dh)
        assert close(cache[:, :, pos0:pos0 + S].transpose(1, 2), want)
        assert (cache[:, :, :pos0] == 5.0).all() and (cache[:, :, pos0 + S:] == 5.0).all()      # nothing else is touched


@pytest.mark.parametrize("V", [1, 5, 4096, 4097, 4100, 32000, 50001, 131072])
def test_argmax_parts_ties_and_special_values(V):
    """One CTA and a cluster of eight per row, vector and scalar loads, parts that are empty or end inside a vector: the lowest
    index of equal maxima wherever they lie, infinities, rows of NaN."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(V)
    rows = [torch.randn(V, device=DEV, generator=gen) for _ in range(9)]
    for i, r in enumerate(rows[:4]):
        at = torch.randint(0, V, (3,), device=DEV, generator=gen)
        r[at] = 7.5 if i < 3 else float("inf")
    rows[4][:] = 1.25
    rows[5][:] = float("-inf")
    rows[6][:] = float("nan")
    rows[7][V // 2:] = float("nan")
    rows[8][V - 1] = 9.0
    lg = torch.stack(rows)
    out = torch.full((9,), -7, dtype=torch.int32, device=DEV)
    tb.k_argmax(lg, out, 9, V)
    torch.cuda.synchronize()
    a = lg.cpu().numpy()
    want = [0 if not np.any(r > -np.inf) else int(np.flatnonzero(r == np.nanmax(r))[0]) for r in a]
    assert out.cpu().tolist() == want


@pytest.mark.parametrize("Dh,Hq,Hkv,TK,kvlen,B", [(64, 4, 4, 16, 1, 1), (64, 8, 2, 16, 16, 2), (128, 8, 1, 32, 17, 1), (64, 16, 8, 64, 33, 3), (128, 4, 2, 16, 65, 1)])
def test_decode_attention_of_short_contexts(Dh, Hq, Hkv, TK, kvlen, B):
    """The automatic choice at contexts of one key to a few chunks (one CTA per head writes the result itself, warps without a
    chunk, chunks that end in a tile's middle) against double precision."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(kvlen)
    nt = (kvlen + TK - 1) // TK
    cfg = replace(KCFG, Dh=Dh, Hq=Hq, Hkv=Hkv, TK=TK, S=kvlen, T=0, B=B, d=Hq * Dh)
    mc = model_cfg(cfg)
    kt, vt = ([torch.randn((B * Hkv * TK, Dh), device=DEV, generator=gen).bfloat16() for _ in range(nt)] for _ in range(2))
    q = torch.randn((B, Hq * Dh), device=DEV, generator=gen).bfloat16()
    o = torch.zeros_like(q)
    scratch = torch.empty(tb.k_attn_scratch_bytes(mc) // 4, dtype=torch.float32, device=DEV)
    tb.k_attn(q, kt, vt, o, mc, B, 1, kvlen - 1, scratch)
    torch.cuda.synchronize()
    K, V = (torch.stack([t.view(B, Hkv, TK, Dh) for t in tiles], dim=2).reshape(B, Hkv, nt * TK, Dh)[:, :, :kvlen].double().repeat_interleave(Hq // Hkv, dim=1) for tiles in (kt, vt))
    p = torch.softmax((K @ q.double().view(B, Hq, Dh, 1)).squeeze(-1) / Dh ** 0.5, dim=-1)
    want = (p.unsqueeze(2) @ V).view(B, Hq * Dh)
    # P counts with 16 bits (2^-16 of averages of V); the result is rounded to bf16: half a step
    assert float(((o.double() - want).abs() - 2.0 ** -8 * want.abs()).max()) < 2.0 ** -14 * float(V.abs().max())


@pytest.mark.parametrize("Dh,Hq,Hkv,TK,kvlen,B", [(64, 32, 8, 64, 9, 16), (64, 16, 2, 64, 130, 8), (128, 32, 8, 128, 17, 8), (128, 8, 8, 16, 40, 8), (128, 8, 1, 64, 700, 5),
                                                  (64, 8, 8, 128, 400, 1)])
def test_decode_attention_of_short_contexts_is_as_exact_as_the_cuda_core_kernels(Dh, Hq, Hkv, TK, kvlen, B):
    """Fewer than 256 chunks of 16 keys in all: P counts with all of its 24 bits.  Of the results, rounded to bf16, hardly any may differ
    from the rounded exact value: fp32 sums of fp32 weights are within 2^-21 of it, so that one in 2^12 lies that close to a
    rounding boundary (2^-21 to either side, of steps of 2^-8); twice that is allowed.  With P rounded to 16 bits it
    is one in 700.  The CUDA-core kernels, forced, meet the same bound."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(kvlen)
    nt = (kvlen + TK - 1) // TK
    cfg = replace(KCFG, Dh=Dh, Hq=Hq, Hkv=Hkv, TK=TK, S=kvlen, T=0, B=B, d=Hq * Dh)
    mc = model_cfg(cfg)
    wrong, total = [0, 0], 0
    for _ in range(8):
        kt, vt = ([torch.randn((B * Hkv * TK, Dh), device=DEV, generator=gen).bfloat16() for _ in range(nt)] for _ in range(2))
        q = torch.randn((B, Hq * Dh), device=DEV, generator=gen).bfloat16()
        scratch = torch.empty(tb.k_attn_scratch_bytes(mc) // 4, dtype=torch.float32, device=DEV)
        K, V = (torch.stack([t.view(B, Hkv, TK, Dh) for t in tiles], dim=2).reshape(B, Hkv, nt * TK, Dh)[:, :, :kvlen].double().repeat_interleave(Hq // Hkv, dim=1) for tiles in (kt, vt))
        p = torch.softmax((K @ q.double().view(B, Hq, Dh, 1)).squeeze(-1) / Dh ** 0.5, dim=-1)
        want = (p.unsqueeze(2) @ V).view(B, Hq * Dh).bfloat16()
        total += want.numel()
        for impl in (0, 1):
            o = torch.zeros_like(q)
            tb.k_attn_decode_select(impl)
            tb.k_attn(q, kt, vt, o, mc, B, 1, kvlen - 1, scratch)
            torch.cuda.synchronize()
            wrong[impl] += int((o != want).sum())
    tb.k_attn_decode_select(0)
    assert max(wrong) <= 2 * total / 2 ** 12, (wrong, total)


@pytest.mark.parametrize("Dh,G,kvlen", [(64, 4, 9), (64, 1, 40), (128, 8, 130), (128, 2, 64)])
def test_decode_attention_of_short_contexts_with_infinities_and_nan(Dh, G, kvlen):
    """An infinity in V reaches the result as it is (not as NaN) where its key has a weight, NaN scores make their row NaN also when they
    are all that one warp sees (its 16 keys)."""
    Hkv, TK, B = 2, 16, 1
    gen = torch.Generator(device=DEV)
    gen.manual_seed(kvlen)
    nt = (kvlen + TK - 1) // TK
    cfg = replace(KCFG, Dh=Dh, Hq=Hkv * G, Hkv=Hkv, TK=TK, S=kvlen, T=0, B=B, d=Hkv * G * Dh)
    mc = model_cfg(cfg)
    kt, vt = ([torch.randn((Hkv * TK, Dh), device=DEV, generator=gen).bfloat16() for _ in range(nt)] for _ in range(2))
    q = torch.randn((B, Hkv * G * Dh), device=DEV, generator=gen).bfloat16()
    scratch = torch.empty(tb.k_attn_scratch_bytes(mc) // 4, dtype=torch.float32, device=DEV)
    vt[0].view(Hkv, TK, Dh)[0, 3, 5] = float("inf")
    vt[0].view(Hkv, TK, Dh)[0, 4, 6] = float("-inf")
    vt[0].view(Hkv, TK, Dh)[0, 3, 7], vt[0].view(Hkv, TK, Dh)[0, 4, 7] = float("inf"), float("-inf")
    o = torch.zeros_like(q)
    tb.k_attn(q, kt, vt, o, mc, B, 1, kvlen - 1, scratch)
    torch.cuda.synchronize()
    got = o.float().view(Hkv, G, Dh)
    assert (got[0, :, 5] == float("inf")).all() and (got[0, :, 6] == float("-inf")).all() and got[0, :, 7].isnan().all()
    rest = [i for i in range(Dh) if i not in (5, 6, 7)]
    assert got[0][:, rest].isfinite().all() and got[1].isfinite().all()
    kt[-1].view(Hkv, TK, Dh)[1] = float("nan")
    tb.k_attn(q, kt, vt, o, mc, B, 1, kvlen - 1, scratch)
    torch.cuda.synchronize()
    assert o.float().view(Hkv, G, Dh)[1].isnan().all()


@pytest.mark.parametrize("M", [9, 16])
def test_row_groups_of_equal_estimates_are_taken_one_at_a_time(M, tmp_path):
    """5120 rows on 148 SMs: three rounds of 12 rows, not two of twice 9."""
    n, K = 5120, 4096
    A, W, C = torch.ones((M, K), device=DEV, dtype=torch.bfloat16), torch.ones((n, K), device=DEV, dtype=torch.bfloat16), torch.zeros((M, n), device=DEV)
    (name, args), = kernels_of(lambda: tb.k_gemm(A, W, C, M, n, K, n, 0, False), tmp_path)
    assert "tgp_wstream_mma_group_kernel" in name and args["shared memory"] == 16 << 10 and bool((C == K).all())


# either side of each line of the dispatch, on 148 SMs: the last length that stays in one CTA (12 chunks of 16 keys for few sequences, more for many),
# the last numbers of (sequence, KV head) pairs that take eight parts (18 of 128 dimensions) and four in clusters (64; 148 in twos)
@pytest.mark.parametrize("Dh,Hq,Hkv,TK,kvlen,B,parts,kernels", [(64, 8, 8, 64, 192, 1, 1, 1), (64, 8, 8, 64, 193, 1, 4, 1), (64, 32, 8, 256, 384, 16, 1, 1), (64, 32, 8, 256, 385, 16, 4, 1),
                                                                (128, 16, 16, 256, 256, 2, 1, 1), (128, 16, 16, 256, 257, 2, 4, 1), (128, 18, 18, 128, 700, 1, 8, 1), (128, 19, 19, 128, 700, 1, 4, 1),
                                                                (128, 32, 8, 256, 2000, 8, 4, 1), (128, 32, 8, 256, 2000, 9, 4, 2), (64, 8, 8, 256, 3000, 24, 3, 2), (64, 8, 8, 4096, 3000, 24, 1, 1)])
def test_parts_of_a_decode_context_on_either_side_of_the_dispatch_lines(Dh, Hq, Hkv, TK, kvlen, B, parts, kernels, tmp_path):
    cfg = replace(KCFG, Dh=Dh, Hq=Hq, Hkv=Hkv, TK=TK, S=kvlen, T=0, B=B, d=Hq * Dh)
    gen = torch.Generator(device=DEV)
    gen.manual_seed(kvlen + B)
    n, G = (kvlen + TK - 1) // TK, Hq // Hkv
    kt, vt = ([torch.randn((B, Hkv, TK, Dh), device=DEV, generator=gen).bfloat16() for _ in range(n)] for _ in range(2))
    q = torch.randn((B, Hkv, G, Dh), device=DEV, generator=gen).bfloat16()
    scratch = torch.zeros(tb.k_attn_scratch_bytes(model_cfg(cfg)) // 4, device=DEV)
    ob = torch.zeros_like(q)
    launched = kernels_of(lambda: tb.k_attn(q, kt, vt, ob, model_cfg(cfg), B, 1, kvlen - 1, scratch), tmp_path)
    assert len(launched) == kernels and launched[0][1]["grid"] == [parts, Hkv, B]
    K, V = (torch.cat(ts, dim=2)[:, :, :kvlen].double() for ts in (kt, vt))
    want = torch.softmax(q.double() @ K.transpose(-1, -2) / Dh ** 0.5, -1) @ V
    # half a bf16 step of the output and of each of the probabilities, whose roundings average out: 2^-9 of the largest V, as in the tests above
    assert float((ob.double() - want).abs().max()) < 2.0 ** -7 * float(want.abs().max()) + 1e-6


# one part, clusters with and without all bits of P, the scratch array; keys that begin a warp's chunks in one of the splits and not in another
@pytest.mark.parametrize("Dh,Hq,Hkv,TK,kvlen,B", [(64, 8, 8, 4096, 400, 1), (64, 4, 4, 64, 64, 1), (64, 32, 8, 128, 700, 1), (128, 32, 8, 1024, 1000, 1),
                                                  (128, 8, 1, 256, 3000, 2), (128, 32, 8, 256, 4000, 4), (64, 16, 2, 64, 40, 2)])
def test_decode_attention_with_keys_of_score_minus_infinity(Dh, Hq, Hkv, TK, kvlen, B):
    """Keys whose scores are -inf (an infinity in K against a negative query) weigh nothing, wherever they lie; a row of nothing else, or with
    one NaN score, is NaN; an infinity in V reaches the result as it is.  As 64 bits have it."""
    cfg = replace(KCFG, Dh=Dh, Hq=Hq, Hkv=Hkv, TK=TK, S=kvlen, T=0, B=B, d=Hq * Dh)
    mc, G, n = model_cfg(cfg), Hq // Hkv, (kvlen + TK - 1) // TK
    gen = torch.Generator(device=DEV)
    gen.manual_seed(kvlen)
    K, V = (torch.zeros((n * TK, B, Hkv, Dh), device=DEV, dtype=torch.bfloat16) for _ in range(2))
    K[:kvlen], V[:kvlen] = (torch.randn((kvlen, B, Hkv, Dh), device=DEV, generator=gen).bfloat16() for _ in range(2))
    q = torch.randn((B, Hq, Dh), device=DEV, generator=gen).bfloat16()
    q[:, :, 0] = -1
    scratch = torch.zeros(tb.k_attn_scratch_bytes(mc) // 4, device=DEV)

    def check(K, V):
        kt, vt = ([t.permute(1, 2, 0, 3).contiguous() for t in T.split(TK)] for T in (K, V))
        ob = torch.zeros((B, Hq, Dh), device=DEV, dtype=torch.bfloat16)
        tb.k_attn(q, kt, vt, ob, mc, B, 1, kvlen - 1, scratch)
        k64, v64 = (T[:kvlen].permute(1, 2, 0, 3).double() for T in (K, V))
        want = (torch.softmax(q.double().view(B, Hkv, G, Dh) @ k64.transpose(-1, -2) / Dh ** 0.5, -1) @ v64).view(B, Hq, Dh)
        got, fin = ob.double(), want.isfinite()
        assert torch.equal(got.isfinite(), fin) and torch.equal(got[~fin].nan_to_num(0.0), want[~fin].nan_to_num(0.0))
        # half a bf16 step of the output and of each of the probabilities, whose roundings average out: 2^-9 of the largest V, as in the tests above
        assert not fin.any() or float((got - want)[fin].abs().max()) < 2.0 ** -7 * float(want[fin].abs().max()) + 1e-6

    for lo, hi in [(0, 16), (16, 32), (0, 32), (64, 80), (kvlen // 32 * 16, kvlen // 32 * 16 + 16), (128, 256), ((kvlen - 1) // 16 * 16, kvlen), (1, kvlen), (0, kvlen)]:
        if lo < kvlen:
            Ki = K.clone()
            Ki[lo:min(hi, kvlen), :, :, 0] = float("inf")
            check(Ki, V)
    for key in (0, kvlen // 2, kvlen - 1):
        Kn, Vi = K.clone(), V.clone()
        Kn[key, B - 1, Hkv - 1] = float("nan")
        check(Kn, V)
        Vi[key, 0, 0, 5], Vi[key, 0, 0, 6] = float("inf"), float("-inf")
        check(K, Vi)


@pytest.mark.parametrize("Dh,S,pos0", [(64, 16, 0), (64, 40, 20), (128, 33, 0), (128, 17, 47)])
def test_attention_of_short_prompts_with_infinities_in_v(Dh, S, pos0):
    """Up to 64 keys what the rounding of P leaves over is multiplied with V too; an infinity in V still reaches the queries that see its
    key as it is, and every other dimension is finite."""
    Hq, Hkv, TK, B = 4, 2, 16, 1
    gen = torch.Generator(device=DEV)
    gen.manual_seed(S)
    nt = (pos0 + S + TK - 1) // TK
    cfg = replace(KCFG, Dh=Dh, Hq=Hq, Hkv=Hkv, TK=TK, S=pos0 + S, T=0, B=B, d=Hq * Dh)
    mc = model_cfg(cfg)
    kt, vt = ([torch.randn((Hkv * TK, Dh), device=DEV, generator=gen).bfloat16() for _ in range(nt)] for _ in range(2))
    q = torch.randn((B * S, Hq * Dh), device=DEV, generator=gen).bfloat16()
    key = 6
    vt[0].view(Hkv, TK, Dh)[0, key, 5], vt[0].view(Hkv, TK, Dh)[0, key, 6] = float("inf"), float("-inf")
    o = torch.zeros_like(q)
    tb.k_attn(q, kt, vt, o, mc, B, S, pos0, None)
    torch.cuda.synchronize()
    got = o.float().view(S, Hq, Dh)
    sees = [i for i in range(S) if pos0 + i >= key]
    assert (got[sees, :2, 5] == float("inf")).all() and (got[sees, :2, 6] == float("-inf")).all()
    assert got[:, :, [i for i in range(Dh) if i not in (5, 6)]].isfinite().all() and got[:, 2:].isfinite().all()


@pytest.mark.parametrize("B,V", [(27, 8192), (27, 8193), (28, 8193), (56, 8196), (112, 12000), (60, 32000), (300, 8200), (300, 24577), (97, 65537)])
def test_argmax_in_eight_four_two_and_one_parts(B, V):
    """Batches and row lengths on either side of the lines between eight parts per row and one; equal maxima in different parts."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(B + V)
    lg = torch.randn((B, V), device=DEV, generator=gen)
    at = torch.randint(0, V, (B, 2), device=DEV, generator=gen)
    lg.scatter_(1, at, 9.0)
    out = torch.full((B,), -7, dtype=torch.int32, device=DEV)
    tb.k_argmax(lg, out, B, V)
    torch.cuda.synchronize()
    assert torch.equal(out.long(), at.min(dim=1).values)


@pytest.mark.parametrize("M,n,K,alone", [(129, 1, 64, True), (200, 1023, 1032, True), (512, 1024, 520, True), (513, 1024, 520, False), (512, 1025, 4096, True), (300, 1025, 4088, False),
                                         (512, 2048, 4104, True), (513, 2048, 4104, False), (256, 2049, 4096, False), (1100, 257, 72, True)])
def test_products_of_few_tiles_alone_have_the_bits_of_the_pairs(M, n, K, alone):
    """More than 128 activation rows on either side of the lines between the one-tile-per-CTA kernel, which a block launched alone takes
    where its tiles are few, and the pairs, which a list takes: the same bits, and the fp64 product."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(M + n + K)
    A = torch.randn((M, K), device=DEV, generator=gen).bfloat16()
    W = (torch.randn((n, K), device=DEV, generator=gen) * 0.02).bfloat16()
    want = A.double() @ W.double().T
    for acc in (False, True):
        c0 = torch.randn((M, n + 4), device=DEV, generator=gen)
        one, pair = c0.clone(), [c0.clone(), c0.clone()]
        tb.k_gemm(A, W, one, M, n, K, n + 4, 0, acc)
        assert tb.k_gemm_last_kernel() == ("tgp_matmul_tc_kernel" if alone else "tgp_matmul_tc_pair_kernel")
        tb.k_gemm_group(A, [W, W], pair, M, [n, n], K, [n + 4, n + 4], acc)
        assert tb.k_gemm_last_kernel() == "tgp_matmul_tc_pair_kernel"
        torch.cuda.synchronize()
        assert tb.k_gemm_status() == 0
        assert torch.equal(one, pair[0]) and torch.equal(one, pair[1]) and torch.equal(one[:, n:], c0[:, n:])
        exact = want + (c0[:, :n].double() if acc else 0)
        assert float((one[:, :n].double() - exact).abs().max()) < 2e-5 * float(exact.abs().max())


# (the first, the sixth and the last two have more tiles than 148 SMs hold clusters of four, so that slices of single CTAs serve them)
@pytest.mark.parametrize("M,n,K", [(129, 4097, 8192), (150, 4096, 8200), (257, 2100, 8192), (509, 2048, 8200), (512, 2048, 14336), (1100, 1000, 8328), (364, 2304, 8192), (236, 3072, 8192), (256, 4600, 8192), (256, 4700, 8192)])
def test_products_of_a_long_k_whose_tiles_two_pairs_share(M, n, K, tmp_path):
    """More than 128 activation rows, K >= 8192 and few tiles: a block alone and in a list of 2 and of 8 (more clusters than fit the GPU at a time) has
    the same bits, no other column changes, and it is as near the fp64 product as fp32 sums are."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(M + n + K)
    A = torch.randn((M, K), device=DEV, generator=gen).bfloat16()
    W = (torch.randn((n, K), device=DEV, generator=gen) * 0.02).bfloat16()
    want = A.double() @ W.double().T
    scratch = torch.empty((M, n), device=DEV)
    (name, args), = kernels_of(lambda: tb.k_gemm(A, W, scratch, M, n, K, n, 0, False), tmp_path)
    tiles = (M + 127) // 128 * ((n + 255) // 256)
    if tiles > 32:
        assert "tgp_wstream_tc_kernel" in name, name
    else:
        assert args["grid"][0] <= 4 * 32, args["grid"]        # also where the tiles are smaller
        assert "tgp_matmul_tc_pair_kernel" in name and ("true" in name or "(bool)1" in name) and args["grid"][0] % 4 == 0, (name, args["grid"])
    for acc in (False, True):
        c0 = torch.randn((M, n + 4), device=DEV, generator=gen)
        one = c0.clone()
        tb.k_gemm(A, W, one, M, n, K, n + 4, 0, acc)
        exact = want + (c0[:, :n].double() if acc else 0)
        for parts in (2, 8):
            C = [c0.clone() for _ in range(parts)]
            tb.k_gemm_group(A, [W] * parts, C, M, [n] * parts, K, [n + 4] * parts, acc)
            torch.cuda.synchronize()
            assert tb.k_gemm_status() == 0
            assert all(torch.equal(one, c) for c in C) and torch.equal(one[:, n:], c0[:, n:])
        # K / 128 additions in each of eight chains, each off by at most a unit of 2^-23 of the running sum (see the real prefill shapes above)
        assert float((one[:, :n].double() - exact).abs().max()) < 2e-5 * max(1.0, K / 8192) * float(exact.abs().max())


@pytest.mark.parametrize("M,n,K", [(129, 4096, 520), (200, 2300, 72), (401, 2048, 1032), (603, 1500, 264), (1030, 1100, 2056)])
def test_products_in_small_tiles_of_pairs_have_the_bits_of_the_largest(M, n, K):
    """Activation rows per tile (16 to 256, by the number of tiles) do not change the sums: the automatic choice and the largest tiles, forced."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(M + n + K)
    A = torch.randn((M, K), device=DEV, generator=gen).bfloat16()
    W = (torch.randn((n, K), device=DEV, generator=gen) * 0.02).bfloat16()
    out = [torch.full((M, n), 7.0, device=DEV) for _ in range(2)]
    tb.k_gemm_group(A, [W, W], [out[0], torch.empty_like(out[0])], M, [n, n], K, [n, n], False)
    tb.k_gemm_tc_variant(3)
    tb.k_gemm(A, W, out[1], M, n, K, n, 0, 0)
    tb.k_gemm_tc_variant(0)
    torch.cuda.synchronize()
    assert tb.k_gemm_status() == 0 and torch.equal(out[0], out[1])
    want = A.double() @ W.double().T
    assert float((out[0].double() - want).abs().max()) < 2e-5 * float(want.abs().max())


@pytest.mark.parametrize("Dh,Hq,Hkv,B,S,pos0,TK", [(64, 4, 4, 1, 384, 0, 64), (128, 4, 1, 2, 500, 0, 128), (64, 8, 2, 1, 129, 300, 64), (128, 2, 2, 3, 201, 1500, 256), (64, 2, 1, 1, 1000, 37, 128)])
def test_prefill_attention_whose_key_blocks_two_ctas_share(Dh, Hq, Hkv, B, S, pos0, TK, tmp_path):
    """Grids that leave SMs idle: two CTAs of a cluster take half of the key blocks each.  Ragged last query blocks, rows whose keys lie in the first half only or begin inside
    the second, scores that grow towards the last keys (a moved exponent reference in one half), against 64 bits; keys of score -inf; an infinity in V, which reaches the rows that see
    its key, whichever half has it, and no row of a query block that ends before the key's block."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(S + pos0)
    n, kv, G = (pos0 + S + TK - 1) // TK, pos0 + S, Hq // Hkv
    cfg = replace(KCFG, Dh=Dh, Hq=Hq, Hkv=Hkv, TK=TK, S=kv, T=0, B=B, d=Hq * Dh)
    mc = model_cfg(cfg)
    q = torch.randn((B, S, Hq, Dh), device=DEV, generator=gen).bfloat16()
    q[..., 0] = 1

    def run(K, V):
        kt, vt = ([t.permute(1, 2, 0, 3).contiguous() for t in T.split(TK)] for T in (K, V))
        ob = torch.zeros((B, S, Hq, Dh), device=DEV, dtype=torch.bfloat16)
        (name, args), = kernels_of(lambda: tb.k_attn(q, kt, vt, ob, mc, B, S, pos0, None), tmp_path)
        assert "tgp_attn_prefill_tc_kernel" in name and args["grid"] == [2 * ((S + 127) // 128), Hq, B], (name, args["grid"])
        assert tb.k_attn_status() == 0
        return ob.double()

    def exact(K, V):
        k64, v64 = (T[:kv].permute(1, 2, 0, 3).double().repeat_interleave(G, 1) for T in (K, V))
        sc = q.permute(0, 2, 1, 3).double() @ k64.transpose(-1, -2) / Dh ** 0.5
        mask = torch.arange(kv, device=DEV)[None, :] > pos0 + torch.arange(S, device=DEV)[:, None]
        return (torch.softmax(sc.masked_fill(mask, -float("inf")), -1) @ v64).permute(0, 2, 1, 3)

    def close(got, want):
        # half a bf16 step of the output and of each of the probabilities, whose roundings average out: 2^-9 of the largest V, as in the tests above
        assert float((got - want).abs().max()) < 2.0 ** -7 * float(want.abs().max()) + 1e-6

    def check(K, V):
        close(run(K, V), exact(K, V))

    K, V = (torch.zeros((n * TK, B, Hkv, Dh), device=DEV, dtype=torch.bfloat16) for _ in range(2))
    K[:kv], V[:kv] = (torch.randn((kv, B, Hkv, Dh), device=DEV, generator=gen).bfloat16() for _ in range(2))
    check(K, V)
    rising = K.clone()                                       # scores up to 150 in units of log2 above the first ones, and falling ones
    rising[:kv, :, :, 0] = (torch.arange(kv, device=DEV)[:, None, None] / kv * 100 * Dh ** 0.5).bfloat16()
    check(rising, V)
    check((-rising.float()).bfloat16(), V)
    hidden = K.clone()                                       # keys of score -inf, the whole first block of the second half among them
    blocks = (kv + 63) // 64
    hidden[64 * ((blocks + 1) // 2):64 * ((blocks + 1) // 2) + 64, :, :, 0] = -float("inf")
    check(hidden, V)
    finite, at = exact(K, V), pos0 + torch.arange(S, device=DEV)
    last = pos0 + torch.clamp((torch.arange(S, device=DEV) // 128 + 1) * 128, max=S) - 1            # position of the last row of a row's query block
    for key in (3, 64 * ((blocks + 1) // 2) - 1, 64 * ((blocks + 1) // 2), kv - 1):                 # the last query block's halves end and begin at the middle two
        Vi = V.clone()
        Vi[key, ..., 5], Vi[key, ..., 6] = float("inf"), -float("inf")
        got, sees, clear = run(K, Vi), at >= key, last // 64 < key // 64
        assert (got[:, sees][..., 5] == float("inf")).all() and (got[:, sees][..., 6] == -float("inf")).all()
        close(got[:, clear], finite[:, clear]) if clear.any() else None
        others = [i for i in range(Dh) if i not in (5, 6)]
        close(got[..., others], finite[..., others])


# a grid whose key blocks two CTAs share and one that leaves no SM idle, both head sizes; mma.sync by length and by choice; the CUDA-core kernels of few queries, of three
# query heads per KV head, of tiles that are no multiple of 16 keys
@pytest.mark.parametrize("Dh,Hq,Hkv,B,S,pos0,TK,impl", [(64, 4, 2, 1, 384, 0, 64, 0), (64, 32, 8, 4, 384, 0, 64, 0), (128, 4, 1, 1, 500, 0, 128, 0), (128, 32, 8, 3, 500, 0, 128, 0),
                                                        (64, 4, 2, 1, 129, 300, 64, 0), (64, 4, 2, 2, 100, 200, 64, 0), (128, 4, 2, 1, 200, 100, 64, 2), (64, 2, 2, 1, 50, 100, 64, 1),
                                                        (64, 4, 2, 2, 5, 120, 64, 0), (64, 3, 1, 2, 1, 170, 64, 0), (128, 4, 2, 1, 1, 170, 24, 0)])
def test_attention_whose_first_keys_score_minus_infinity(Dh, Hq, Hkv, B, S, pos0, TK, impl):
    """The first keys of every row, or all that a row sees, score -inf: they weigh nothing, and a row of nothing else is NaN, whichever kernel the grid, the number of
    queries or the tiles choose.  As 64 bits have it."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(S + pos0 + Dh)
    n, kv, G = (pos0 + S + TK - 1) // TK, pos0 + S, Hq // Hkv
    cfg = replace(KCFG, Dh=Dh, Hq=Hq, Hkv=Hkv, TK=TK, S=kv, T=0, B=B, d=Hq * Dh)
    mc = model_cfg(cfg)
    q = torch.randn((B, S, Hq, Dh), device=DEV, generator=gen).bfloat16()
    q[..., 0] = 1
    K, V = (torch.zeros((n * TK, B, Hkv, Dh), device=DEV, dtype=torch.bfloat16) for _ in range(2))
    K[:kv], V[:kv] = (torch.randn((kv, B, Hkv, Dh), device=DEV, generator=gen).bfloat16() for _ in range(2))
    scratch = torch.zeros(tb.k_attn_scratch_bytes(mc) // 4, device=DEV) if S == 1 else None
    mask = torch.arange(kv, device=DEV)[None, :] > pos0 + torch.arange(S, device=DEV)[:, None]
    for lo, hi in ((0, 16), (0, 33), (0, 64), (0, 128), (64, 160), (0, kv)):
        hidden = K.clone()
        hidden[lo:min(hi, kv), :, :, 0] = -float("inf")
        kt, vt = ([t.permute(1, 2, 0, 3).contiguous() for t in T.split(TK)] for T in (hidden, V))
        ob = torch.zeros((B, S, Hq, Dh), device=DEV, dtype=torch.bfloat16)
        tb.k_attn_select(impl)
        tb.k_attn(q, kt, vt, ob, mc, B, S, pos0, scratch)
        tb.k_attn_select(0)
        torch.cuda.synchronize()
        assert tb.k_attn_status() == 0
        k64, v64 = (T[:kv].permute(1, 2, 0, 3).double().repeat_interleave(G, 1) for T in (hidden, V))
        sc = q.permute(0, 2, 1, 3).double() @ k64.transpose(-1, -2) / Dh ** 0.5
        want = (torch.softmax(sc.masked_fill(mask, -float("inf")), -1) @ v64).permute(0, 2, 1, 3)
        got, fin = ob.double(), want.isfinite()
        assert torch.equal(got.isfinite(), fin), (lo, hi)
        # half a bf16 step of the output and of each of the probabilities, whose roundings average out: 2^-9 of the largest V, as in the tests above
        assert not fin.any() or float((got - want)[fin].abs().max()) < 2.0 ** -7 * float(want[fin].abs().max()) + 1e-6


def test_products_whose_tiles_two_pairs_share_give_up_on_a_wait_that_runs_out_and_recover():
    """The four CTAs of the first cluster never load their second stage: the waits for their tile run out in both pairs, none of the four stores anything, every other
    tile is right, and the next launch is correct."""
    M, n, K = 509, 2048, 8192
    gen = torch.Generator(device=DEV)
    gen.manual_seed(5)
    A = torch.randn((M, K), device=DEV, generator=gen).bfloat16()
    W = (torch.randn((n, K), device=DEV, generator=gen) * 0.02).bfloat16()
    want = A.double() @ W.double().T
    SENT = 12345.0
    tb.k_status_clear()
    try:
        tb.k_wait_test(2_000_000, 1)
        C = torch.full((M, n), SENT, device=DEV)
        tb.k_gemm(A, W, C, M, n, K, n, 0, 0)
        torch.cuda.synchronize()
        assert tb.k_gemm_status() >> 8 in (2, 3)              # the MMA threads' waits for the stage, the epilogues' for the accumulators
        untouched = C == SENT
        rows = int(untouched[:, 0].sum())                     # (the tile's activation rows)
        assert 32 <= rows <= 128 and rows % 32 == 0 and untouched[:rows, :256].all() and int(untouched.sum()) == 256 * rows
        assert float((C.double() - want)[~untouched].abs().max()) < 2e-5 * float(want.abs().max())
    finally:
        tb.k_wait_test(0, -1)
        tb.k_status_clear()
    tb.k_gemm(A, W, C, M, n, K, n, 0, 0)
    torch.cuda.synchronize()
    assert tb.k_gemm_status() == 0 and float((C.double() - want).abs().max()) < 2e-5 * float(want.abs().max())


@pytest.mark.parametrize("Dh", [64, 128])
def test_attention_whose_key_blocks_two_ctas_share_gives_up_on_a_wait_that_runs_out_and_recovers(Dh):
    """The grid's first CTA - the first half of the key blocks of the last 128 queries of head 0 - never loads its second V block: its waits run out, neither it nor the CTA
    that has the other half stores anything, all other rows are right, and the next launch is correct."""
    S, Hq, Hkv, TK = 512, 4, 2, 64
    cfg = replace(KCFG, Dh=Dh, Hq=Hq, Hkv=Hkv, TK=TK, S=S, T=0, B=1, d=Hq * Dh)
    mc = model_cfg(cfg)
    gen = torch.Generator(device=DEV)
    gen.manual_seed(Dh)
    q, K, V = (torch.randn((S, h, Dh), device=DEV, generator=gen).bfloat16() for h in (Hq, Hkv, Hkv))
    kt, vt = ([t.permute(1, 0, 2).contiguous()[None] for t in T.split(TK)] for T in (K, V))
    k64, v64 = (T.permute(1, 0, 2).double().repeat_interleave(Hq // Hkv, 0) for T in (K, V))
    sc = (q.permute(1, 0, 2).double() @ k64.transpose(-1, -2) / Dh ** 0.5).masked_fill(torch.ones((S, S), device=DEV, dtype=torch.bool).triu(1), -float("inf"))
    want = (torch.softmax(sc, -1) @ v64).permute(1, 0, 2)
    tol = 2.0 ** -7 * float(want.abs().max()) + 1e-6          # as in the tests above
    tb.k_status_clear()
    try:
        tb.k_wait_test(2_000_000, 1)
        ob = torch.full((S, Hq, Dh), 768.0, dtype=torch.bfloat16, device=DEV)
        tb.k_attn(q, kt, vt, ob, mc, 1, S, 0, None)
        torch.cuda.synchronize()
        assert tb.k_attn_status() in (1, 2, 3)
        untouched = ob == 768.0
        assert untouched[S - 128:, 0].all() and int(untouched.sum()) == 128 * Dh
        assert float((ob.double() - want)[~untouched].abs().max()) < tol
    finally:
        tb.k_wait_test(0, -1)
        tb.k_status_clear()
    tb.k_attn(q, kt, vt, ob, mc, 1, S, 0, None)
    torch.cuda.synchronize()
    assert tb.k_attn_status() == 0 and float((ob.double() - want).abs().max()) < tol


# on either side of the lines: a third, a half and all of 148 SMs have a CTA
@pytest.mark.parametrize("Dh,Hq,B,S,blocks,two", [(64, 12, 1, 500, 5, False), (64, 12, 1, 384, 6, True), (128, 16, 1, 300, 7, False), (128, 16, 1, 300, 8, True), (64, 16, 1, 500, 7, False),
                                                  (64, 18, 1, 500, 8, True), (128, 16, 1, 500, 9, False), (128, 18, 1, 500, 10, True), (64, 19, 1, 500, 11, False), (64, 16, 3, 380, 12, True),
                                                  (128, 19, 1, 500, 13, False), (128, 37, 1, 500, 14, True), (64, 38, 1, 500, 20, False)])
def test_key_blocks_are_shared_where_that_is_faster(Dh, Hq, B, S, blocks, two, tmp_path):
    kv, TK = 64 * blocks - 10, 128
    n, pos0 = (kv + TK - 1) // TK, 64 * blocks - 10 - S
    if pos0 < 0:
        pos0, S = 0, kv
    mc = model_cfg(replace(KCFG, Dh=Dh, Hq=Hq, Hkv=Hq, TK=TK, S=kv, T=0, B=B, d=Hq * Dh))
    q = torch.randn((B, S, Hq, Dh), device=DEV).bfloat16()
    kt, vt = ([torch.randn((B, Hq, TK, Dh), device=DEV).bfloat16() for _ in range(n)] for _ in range(2))
    ob = torch.empty_like(q)
    (name, args), = kernels_of(lambda: tb.k_attn(q, kt, vt, ob, mc, B, S, pos0, None), tmp_path)
    assert "tgp_attn_prefill_tc_kernel" in name and args["grid"] == [(2 if two else 1) * ((S + 127) // 128), Hq, B], (name, args["grid"])
