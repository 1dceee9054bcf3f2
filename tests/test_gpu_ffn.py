"""GPU parity of hidden RMSNorm, fused residual + RMSNorm, SwiGLU and the dense linear layer
against the CPU oracle, and their bit-identity between batched and row-by-row use (the paper's
operator table verifies each of them bitwise between full-sequence and token-wise execution)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

import oracle
from paper_2609_35140_b200 import build as tik_build
from gpu_common import BAND, NARROW, PAIR_UNITS, UNITS, count_diff, linear_schedule

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tik():
    from paper_2609_35140_b200 import binding
    binding.load()
    yield binding
    assert binding.device_status() == 0


def _randn(shape, seed, std=1.0):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return (torch.randn(shape, generator=g, device="cuda") * std).to(torch.bfloat16)


def _close_bf16(got, ref, abs_tol=1e-6):
    g = got.float().cpu().numpy().astype(np.float64)
    assert np.all(np.abs(g - ref) <= 2.0 ** -8 * np.abs(ref) + abs_tol), float(np.abs(g - ref).max())


def _schedule(tik, T, K, N):
    return linear_schedule(tik.load(), T, K, N, torch.cuda.get_device_properties(0).multi_processor_count)[0]


def _band_rows(tik, x, W):
    """tik_linear(x, W) as part of a call that runs as CTA pairs in the band raster, whatever kernel a call of x and W
    alone takes: more rows of x and more weight rows (both repeated) leave a row's and a column's result alone."""
    (T, K), N = x.shape, W.shape[0]
    rows, cols = max(T, 2049), max(N, 512)
    assert _schedule(tik, rows, K, cols) == BAND
    xs, Ws = x.repeat(-(-rows // T), 1)[:rows].contiguous(), W.repeat(-(-cols // N), 1)[:cols].contiguous()
    return tik.tik_linear(xs, Ws)[:T, :N].contiguous()


@pytest.mark.parametrize("H", [8, 64, 1000, 1536, 3584, 4096, 5120, 8192])
def test_rmsnorm_matches_oracle_and_rows_are_independent(tik, H):
    T = 37
    x = _randn((T, H), 500 + H, 2.0)
    w = (1 + 0.2 * _randn((H,), 600 + H).float()).to(torch.bfloat16)
    y = tik.tik_rmsnorm(x, w, 1e-6)
    _close_bf16(y, oracle.rmsnorm(x.float().cpu().numpy(), w.float().cpu().numpy(), 1e-6))
    for a, b in [(0, 1), (5, 6), (30, 37)]:
        assert count_diff(tik.tik_rmsnorm(x[a:b].contiguous(), w, 1e-6), y[a:b]) == 0
    # in place
    x2 = x.clone()
    tik.tik_rmsnorm(x2, w, 1e-6, y=x2)
    assert count_diff(x2, y) == 0


@pytest.mark.parametrize("H", [64, 1536, 4096, 8192])
def test_fused_residual_rmsnorm(tik, H):
    T = 29
    x = _randn((T, H), 700 + H)
    res0 = _randn((T, H), 800 + H, 20.0)
    w = (1 + 0.2 * _randn((H,), 900 + H).float()).to(torch.bfloat16)
    res = res0.clone()
    y = tik.tik_rmsnorm(x, w, 1e-6, residual=res)
    y_ref, s_ref = oracle.rmsnorm(x.float().cpu().numpy(), w.float().cpu().numpy(), 1e-6,
                                  residual=res0.float().cpu().numpy())
    assert np.array_equal(res.float().cpu().numpy(), s_ref)         # the stored sum, bit for bit
    assert count_diff(res, x + res0) == 0                           # == a bf16 tensor add
    _close_bf16(y, y_ref)
    assert count_diff(y, tik.tik_rmsnorm(res, w, 1e-6)) == 0        # fused == add, then plain norm
    # token-wise == batched
    r1 = res0[3:4].clone()
    y1 = tik.tik_rmsnorm(x[3:4].contiguous(), w, 1e-6, residual=r1)
    assert count_diff(y1, y[3:4]) == 0 and count_diff(r1, res[3:4]) == 0


@pytest.mark.parametrize("T,I", [(1, 8), (33, 1000), (257, 8960), (64, 18944), (1100, 8960)])   # the last one: four vectors per thread, ragged last block
def test_swiglu(tik, T, I):
    gu = _randn((T, 2 * I), 1000 + I, 3.0)
    gu[0, :4] = torch.tensor([0.0, 40.0, -40.0, -100.0], dtype=torch.bfloat16)
    out = tik.tik_swiglu(gu)
    _close_bf16(out, oracle.swiglu(gu.float().cpu().numpy()), abs_tol=1e-5)
    assert bool(torch.isfinite(out).all())
    t = T // 2
    assert count_diff(tik.tik_swiglu(gu[t:t + 1].contiguous()), out[t:t + 1]) == 0


@pytest.mark.parametrize("T,K,N", [(1, 64, 8), (300, 1536, 1000), (129, 8960, 1536), (700, 1536, 2304),
                                   (4100, 256, 1032)])
def test_linear_matches_oracle_and_is_batch_invariant(tik, T, K, N):
    x = _randn((T, K), 1100 + K)
    W = _randn((N, K), 1200 + N, 0.02)
    y = tik.tik_linear(x, W)
    ref = oracle.linear(x.float().cpu().numpy(), W.float().cpu().numpy())
    g = y.float().cpu().numpy().astype(np.float64)
    scale = 0.02 * np.sqrt(K)
    assert np.all(np.abs(g - ref) <= 2.0 ** -8 * np.abs(ref) + 1e-4 * scale), float(np.abs(g - ref).max())
    # a row alone (decode), a ragged slice and a slice that starts inside a 128-row tile
    for a, b in [(0, 1), (T - 1, T), (T // 3, T // 3 + 5), (max(0, T - 131), T)]:
        if a < b:
            assert count_diff(tik.tik_linear(x[a:b].contiguous(), W), y[a:b]) == 0, (a, b)
    # canary: nothing is written outside [T][N]
    buf = torch.full((T + 2, N), -7.0, dtype=torch.bfloat16, device="cuda")
    tik.tik_linear(x, W, y=buf[1:T + 1])
    assert bool((buf[0] == -7.0).all()) and bool((buf[T + 1] == -7.0).all())
    assert count_diff(buf[1:T + 1], y) == 0


@pytest.mark.parametrize("K,N", [(512, 37888), (256, 55296), (1024, 5120), (192, 1000), (128, 72), (64, 40000),
                                 (27648, 5120), (3584, 37888)])
def test_decode_shaped_linear_equals_rows_of_a_batched_call(tik, K, N):
    """Calls of one and two row tiles, by the narrow schedule or over units of 64, 128 or 256 columns with 32, 64 or
    128 staged rows or over pairs' units: each returns the bits of the same rows inside a 300-row call, which are
    those of the band raster (CTA pairs, 256-column steps), and writes nothing outside its [T][N] block."""
    x = _randn((300, K), 2100 + K)
    W = _randn((N, K), 2200 + N % 977, 0.02)
    y = tik.tik_linear(x, W)
    assert count_diff(y, _band_rows(tik, x, W)) == 0
    ncol = min(N, 4096)                   # the oracle on three rows and the first columns (full-size K x N: seconds)
    ref = oracle.linear(x[:3].float().cpu().numpy(), W[:ncol].float().cpu().numpy())
    g = y[:3, :ncol].float().cpu().numpy().astype(np.float64)
    assert np.all(np.abs(g - ref) <= 2.0 ** -8 * np.abs(ref) + 1e-4 * 0.02 * np.sqrt(K))
    for a, T in [(0, 1), (7, 16), (100, 32), (3, 33), (50, 64), (171, 65), (172, 128), (90, 129), (20, 200), (44, 256)]:
        buf = torch.full((T + 2, N), -7.0, dtype=torch.bfloat16, device="cuda")
        tik.tik_linear(x[a:a + T].contiguous(), W, y=buf[1:T + 1])
        assert count_diff(buf[1:T + 1], y[a:a + T]) == 0, (a, T)
        assert bool((buf[0] == -7.0).all()) and bool((buf[T + 1] == -7.0).all())
    assert tik.device_status() == 0


def test_ffn_block_composition(tik):
    """norm -> gate/up projection -> SwiGLU -> down projection, batched and token by token."""
    T, H, I = 70, 512, 1408
    x = _randn((T, H), 1)
    res = _randn((T, H), 2)
    w = (1 + 0.1 * _randn((H,), 3).float()).to(torch.bfloat16)
    Wgu, Wd = _randn((2 * I, H), 4, 0.03), _randn((H, I), 5, 0.03)

    def block(xs, rs):
        r = rs.clone()
        h = tik.tik_rmsnorm(xs, w, 1e-6, residual=r)
        return tik.tik_linear(tik.tik_swiglu(tik.tik_linear(h, Wgu)), Wd), r

    y, r = block(x, res)
    for t in (0, 17, 69):
        y1, r1 = block(x[t:t + 1].contiguous(), res[t:t + 1].contiguous())
        assert count_diff(y1, y[t:t + 1]) == 0 and count_diff(r1, r[t:t + 1]) == 0
    # against the oracle chain evaluated on the GPU's own intermediate roundings
    h_ref, s = oracle.rmsnorm(x.float().cpu().numpy(), w.float().cpu().numpy(), 1e-6, residual=res.float().cpu().numpy())
    h = tik.tik_rmsnorm(x, w, 1e-6, residual=res.clone())
    _close_bf16(h, h_ref)
    gu = tik.tik_linear(h, Wgu)
    a = tik.tik_swiglu(gu)
    _close_bf16(a, oracle.swiglu(gu.float().cpu().numpy()), abs_tol=1e-5)
    ref = oracle.linear(a.float().cpu().numpy(), Wd.float().cpu().numpy())
    g = y.float().cpu().numpy().astype(np.float64)
    assert np.all(np.abs(g - ref) <= 2.0 ** -8 * np.abs(ref) + 1e-3)


def test_ffn_invalid_arguments(tik):
    x = _randn((4, 64), 1)
    w = _randn((64,), 2)
    with pytest.raises(tik.TikError):
        tik.tik_rmsnorm(_randn((4, 12), 1), _randn((12,), 2), 1e-6)          # H % 8
    with pytest.raises(tik.TikError):
        tik.tik_rmsnorm(x, w, -1.0)
    with pytest.raises(tik.TikError):
        tik.tik_linear(_randn((4, 32), 1), _randn((8, 32), 2))                # K % 64
    with pytest.raises(tik.TikError):
        tik.tik_linear(x, _randn((12, 64), 2))                                # N % 8
    with pytest.raises(tik.TikError):
        tik.tik_swiglu(_randn((4, 24), 1))                                    # I % 8
    assert tik.tik_linear(x[:0], _randn((8, 64), 2)).shape == (0, 8)


@pytest.mark.parametrize("K,N", [(64, 8), (576, 1184), (576, 1192), (4096, 1536), (1024, 3584), (320, 9472), (256, 9480)])
def test_narrow_linear_equals_rows_of_a_batched_call(tik, K, N):
    """T <= 80 and N <= 64 columns per SM: weights as the M operand, 8 .. 64 rows of them per CTA.  Row counts
    around the multiples of 16 that are staged, K tails of a ring stage, outputs of one CTA, of whole and ragged
    last CTAs, and the first N beyond the range: the bits of a batched call, which are those of the band raster (a
    300-row call of few columns is narrow too), nothing written outside y."""
    x = _randn((300, K), 3100 + K)
    W = _randn((N, K), 3200 + N % 977, 0.02)
    y = tik.tik_linear(x, W)
    assert count_diff(y, _band_rows(tik, x, W)) == 0
    assert {_schedule(tik, T, K, N) for T in (1, 16, 80)} == {NARROW if N <= 9472 else UNITS}
    ref = oracle.linear(x[:3].float().cpu().numpy(), W.float().cpu().numpy())
    g = y[:3].float().cpu().numpy().astype(np.float64)
    assert np.all(np.abs(g - ref) <= 2.0 ** -8 * np.abs(ref) + 1e-4 * 0.02 * np.sqrt(K))
    for a, T in [(0, 1), (5, 15), (7, 16), (9, 17), (100, 32), (3, 48), (50, 65), (171, 80), (160, 81), (172, 97)]:
        buf = torch.full((T + 2, N), -7.0, dtype=torch.bfloat16, device="cuda")
        tik.tik_linear(x[a:a + T].contiguous(), W, y=buf[1:T + 1])
        assert count_diff(buf[1:T + 1], y[a:a + T]) == 0, (a, T)
        assert bool((buf[0] == -7.0).all()) and bool((buf[T + 1] == -7.0).all())
    assert tik.device_status() == 0


@pytest.mark.parametrize("K,N", [(64, 8), (192, 1000), (576, 1536), (320, 9480), (128, 37888)])
def test_mid_size_linear_equals_rows_of_a_batched_call(tik, K, N):
    """2 .. 16 row tiles: the narrow schedule, single CTAs over units of 64, 128 or 256 columns x one row tile, or
    pairs, by rules that reach each of them at these sizes.  Row counts around the tiles and around the range's ends:
    the bits of a longer call, which are those of the band raster, nothing written outside y."""
    x = _randn((2300, K), 3300 + K)
    W = _randn((N, K), 3400 + N % 977, 0.02)
    y = tik.tik_linear(x, W)
    assert count_diff(y, _band_rows(tik, x, W)) == 0
    kinds = {_schedule(tik, T, K, N) for T in (129, 256, 385, 768, 1500, 2048)}
    assert kinds == {8: {NARROW}, 1000: {NARROW, UNITS}, 1536: {NARROW, UNITS}, 9480: {UNITS, PAIR_UNITS},
                     37888: {UNITS, PAIR_UNITS}}[N]
    rows = [0, 1150, 2299]
    ref = oracle.linear(x[rows].float().cpu().numpy(), W.float().cpu().numpy())
    g = y[rows].float().cpu().numpy().astype(np.float64)
    assert np.all(np.abs(g - ref) <= 2.0 ** -8 * np.abs(ref) + 1e-4 * 0.02 * np.sqrt(K))
    for a, T in [(0, 129), (7, 255), (130, 256), (9, 257), (3, 385), (500, 768), (77, 1025), (1, 1500), (128, 2047), (252, 2048), (5, 2049)]:
        buf = torch.full((T + 2, N), -7.0, dtype=torch.bfloat16, device="cuda")
        tik.tik_linear(x[a:a + T].contiguous(), W, y=buf[1:T + 1])
        assert count_diff(buf[1:T + 1], y[a:a + T]) == 0, (a, T)
        assert bool((buf[0] == -7.0).all()) and bool((buf[T + 1] == -7.0).all())
    assert tik.device_status() == 0


@pytest.mark.parametrize("K,N", [(64, 256), (576, 1536), (640, 4608), (192, 6000)])
def test_narrow_linear_with_x_as_the_m_operand(tik, K, N):
    """Row counts where x becomes the M operand of the narrow schedule (M64, M128, tiles of 128 rows), around the
    8-row atoms and the tiles: the bits of a batched call, which are those of the band raster and near the
    oracle's, nothing written outside y."""
    x = _randn((2300, K), 3500 + K)
    W = _randn((N, K), 3600 + N % 977, 0.02)
    y = tik.tik_linear(x, W)
    assert count_diff(y, _band_rows(tik, x, W)) == 0
    assert _schedule(tik, 72, K, N) == NARROW and _schedule(tik, 127, K, N) == NARROW
    rows = [0, 700, 2299]
    ref = oracle.linear(x[rows].float().cpu().numpy(), W.float().cpu().numpy())
    g = y[rows].float().cpu().numpy().astype(np.float64)
    assert np.all(np.abs(g - ref) <= 2.0 ** -8 * np.abs(ref) + 1e-4 * 0.02 * np.sqrt(K))
    for a, T in [(0, 17), (5, 24), (9, 40), (3, 41), (100, 63), (50, 64), (172, 65), (1, 72), (7, 88), (11, 127), (64, 128), (13, 129), (700, 260)]:
        buf = torch.full((T + 2, N), -7.0, dtype=torch.bfloat16, device="cuda")
        tik.tik_linear(x[a:a + T].contiguous(), W, y=buf[1:T + 1])
        assert count_diff(buf[1:T + 1], y[a:a + T]) == 0, (a, T)
        assert bool((buf[0] == -7.0).all()) and bool((buf[T + 1] == -7.0).all())
    assert tik.device_status() == 0


@pytest.mark.parametrize("T,K,N", [(768, 320, 1152), (768, 320, 1184), (384, 192, 1576), (2304, 128, 256), (3456, 128, 256),
                                   (5000, 64, 128), (18944, 64, 40), (20000, 128, 8), (20000, 64, 24)])
def test_narrow_linear_at_the_ends_of_its_range(tik, T, K, N):
    """As many CTAs as SMs, one more (another kernel takes the call), more than 16 row tiles, and more row tiles than
    SMs with one CTA each: the bits of the band raster, nothing written outside y."""
    x = _randn((T, K), 3700 + K)
    W = _randn((N, K), 3800 + N % 977, 0.02)
    narrow = (T, N) not in ((768, 1184), (3456, 256))
    assert (_schedule(tik, T, K, N) == NARROW) == narrow
    buf = torch.full((T + 2, N), -7.0, dtype=torch.bfloat16, device="cuda")
    tik.tik_linear(x, W, y=buf[1:T + 1])
    assert count_diff(buf[1:T + 1], _band_rows(tik, x, W)) == 0
    assert bool((buf[0] == -7.0).all()) and bool((buf[T + 1] == -7.0).all())
    assert tik.device_status() == 0


@pytest.mark.parametrize("K,N", [(64, 9480), (576, 12288), (1024, 24576), (256, 40000)])
def test_unit_linear_of_a_few_rows(tik, K, N):
    """Column units of 128, 256 and 128 columns with 8, 16 or 32 staged rows of x, fewer than an MMA spans: the bits of
    the band raster, nothing written outside y, and rows of infinities in W stay in their own columns."""
    x = _randn((40, K), 3900 + K)
    W = _randn((N, K), 4000 + N % 977, 0.02)
    y = _band_rows(tik, x, W)
    W2 = W.clone()
    W2[5], W2[70] = float("inf"), float("nan")           # (what the MMA reads behind the staged rows is W)
    keep = torch.ones(N, dtype=torch.bool, device="cuda")
    keep[5] = keep[70] = False
    for a, T in [(0, 1), (3, 2), (9, 7), (30, 8), (4, 9), (20, 15), (24, 16), (1, 17), (8, 32)]:
        assert _schedule(tik, T, K, N) == UNITS
        buf = torch.full((T + 2, N), -7.0, dtype=torch.bfloat16, device="cuda")
        tik.tik_linear(x[a:a + T].contiguous(), W, y=buf[1:T + 1])
        assert count_diff(buf[1:T + 1], y[a:a + T]) == 0, (a, T)
        assert bool((buf[0] == -7.0).all()) and bool((buf[T + 1] == -7.0).all())
        assert count_diff(tik.tik_linear(x[a:a + T].contiguous(), W2)[:, keep], y[a:a + T][:, keep]) == 0, (a, T)
    assert tik.device_status() == 0


@pytest.mark.parametrize("rows,I", [(1, 8), (513, 8), (5, 264), (3, 2056), (700, 12000), (1049000, 8)])
def test_swiglu_gates_of_every_size(tik, rows, I):
    """Rows of less than a block's vectors, of more, and a last block that ends in the middle; gates from those whose
    reciprocal is subnormal to those whose weight is one, infinities and NaN.  One bf16 rounding (2^-9) and fp32
    arithmetic below it.  Where 2^(-g log2 e) is beyond fp32 (g < -88.72) the weight is 0: off by at most
    88.73 * 2^-128 * 7 < 1.9e-36, the most that |g| e^g u comes to there (u <= 7)."""
    g = torch.linspace(-104.0, 104.0, rows * I, device="cuda").to(torch.bfloat16)
    special = torch.tensor([float("inf"), float("-inf"), float("nan"), 0.0, -87.5, -88.5, -90.0, 88.5], device="cuda")
    g[:8] = special.to(torch.bfloat16)
    u = (1.0 + torch.arange(rows * I, device="cuda") % 7).to(torch.bfloat16)
    got = tik.tik_swiglu(torch.cat([g.view(rows, I), u.view(rows, I)], dim=1).contiguous()).view(-1).double()
    want = g.double() / (1.0 + torch.exp(-g.double())) * u.double()
    odd = ~torch.isfinite(want)
    assert torch.equal(torch.nan_to_num(got[odd], nan=7.0), torch.nan_to_num(want[odd], nan=7.0))
    assert bool(((got - want).abs()[~odd] <= 2.0 ** -8 * want.abs()[~odd] + 1.9e-36).all())


@pytest.fixture(scope="module")
def swiglu_check(tmp_path_factory):
    """tests/swiglu_check.cu, built with the library's flags against the library's header."""
    out = str(tmp_path_factory.mktemp("swiglu") / "swiglu_check.so")
    source = os.path.join(os.path.dirname(os.path.abspath(__file__)), "swiglu_check.cu")
    r = subprocess.run([tik_build._nvcc()] + tik_build.NVCC_FLAGS + ["-I" + tik_build.CSRC, "-shared", source, "-o", out],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    lib = ctypes.CDLL(out)
    lib.swiglu_check_rcp.argtypes = [ctypes.c_uint, ctypes.c_uint, ctypes.c_void_p]
    lib.swiglu_check_gates.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_void_p]
    return lib


def _float_bits(x):
    return int(np.float32(x).view(np.uint32))


def test_swiglu_reciprocal_is_the_correctly_rounded_one(swiglu_check):
    """Every float from 1 to 2^126, in both lanes.  The approximate reciprocal alone is not that one everywhere."""
    first, last = _float_bits(1.0), _float_bits(2.0 ** 126)
    count = torch.zeros(3, dtype=torch.int64, device="cuda")
    assert swiglu_check.swiglu_check_rcp(first, last, count.data_ptr()) == 0
    differ, approx, seen = count.tolist()
    assert seen == last - first + 1 and approx > 0
    assert differ == 0


def test_swiglu_two_at_a_time_has_the_bits_of_one_at_a_time(swiglu_check):
    """All 65536 bf16 gates, infinities and NaN among them, beside a gate of another size."""
    up = torch.tensor([1.0, -1.0, 0.0, 3.0, -0.1, 1e-38, 3e38, float("inf"), float("nan")], device="cuda").to(torch.bfloat16).float()
    count = torch.zeros(3, dtype=torch.int64, device="cuda")
    assert swiglu_check.swiglu_check_gates(up.data_ptr(), up.numel(), count.data_ptr()) == 0
    assert count[2].item() == 65536
    assert count[0].item() == 0


@pytest.mark.parametrize("rows,I", [(33000, 264), (4200, 2040), (8200, 1032), (70000, 120), (12000, 704)])
def test_swiglu_rows_of_less_than_a_block_in_large_calls(tik, rows, I):
    """Calls of four vectors per thread whose rows have 15 .. 255 vectors: a step of 256 is dt whole rows and dc vectors,
    both above zero, with and without a carry, and a last block that ends in the middle.  The bits of the same rows in
    calls of one vector per thread."""
    vpr = I // 8
    assert rows * vpr >= 1 << 20 and rows * vpr % 1024 and 256 // vpr and 256 % vpr
    gu = _randn((rows, 2 * I), 1400 + I, 3.0)
    out = torch.full((rows + 1, I), -7.0, dtype=torch.bfloat16, device="cuda")
    tik.tik_swiglu(gu, out=out[:rows])
    small = (1 << 20) // vpr - 1
    for a in range(0, rows, small):
        part = gu[a:a + small]
        assert part.shape[0] * vpr < 1 << 20
        assert count_diff(tik.tik_swiglu(part), out[a:min(a + small, rows)]) == 0, a
    assert bool((out[rows] == -7.0).all())
    g, u = gu[:, :I].double(), gu[:, I:].double()
    want = g / (1.0 + torch.exp(-g)) * u
    assert bool(((out[:rows].double() - want).abs() <= 2.0 ** -8 * want.abs() + 1e-6).all())
