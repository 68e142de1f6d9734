"""Kernels at the sizes where they can go wrong: edges of tiles, remainders, the smallest and largest of a dispatch's range,
against the CPU oracle."""
import numpy as np
import pytest
import torch

import synth_inputs as si
from oracle import goq_oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def goq():
    from paper_2605_26092_b200 import build
    build.build()
    from paper_2605_26092_b200 import goq as g
    g.lib()
    assert torch.cuda.is_available()
    return g


def _unaligned(a, shift):
    """The array on the device, `shift` elements behind an aligned address."""
    t = torch.from_numpy(np.ascontiguousarray(a))
    buf = torch.empty(t.numel() + shift, dtype=t.dtype, device="cuda")
    buf[shift:] = t.reshape(-1).cuda()
    return buf[shift:]


@pytest.mark.parametrize("b", [2, 3, 4])
@pytest.mark.parametrize("n,k,g,shift", [(1, 8, 8, 0), (16, 128, 128, 0), (17, 136, 8, 0), (15, 240, 16, 3), (33, 384, 64, 1), (40, 96, 32, 0)])
def test_pack_edges(goq, n, k, g, b, shift):
    """Rows and columns that end inside a record, code and record arrays at odd addresses: the fields come back unchanged."""
    rng = np.random.default_rng(n + k + b)
    codes = rng.integers(0, 1 << b, size=(n, k), dtype=np.uint8)
    meta = rng.integers(0, 64, size=(n, k // 8), dtype=np.uint8)
    coef = rng.standard_normal((n, k // g, 2)).astype(np.float16)
    d = goq.desc(n, k, g, b)
    packed = torch.full((goq.packed_bytes(d),), 0xA5, dtype=torch.uint8, device="cuda")
    goq.pack(d, _unaligned(codes, shift), _unaligned(meta, shift), _unaligned(coef.view(np.int16), shift), packed)
    b1 = torch.empty((n, k), dtype=torch.uint8, device="cuda")
    b2 = torch.empty((n, k), dtype=torch.uint8, device="cuda")
    cf = torch.empty((n, k // g, 2), dtype=torch.int16, device="cuda")
    goq.unpack(d, packed, b1, b2, cf)
    torch.cuda.synchronize()
    assert np.array_equal(b1.cpu().numpy(), codes)
    assert np.array_equal(cf.cpu().numpy().view(np.uint16), coef.view(np.uint16))
    ref = O.decode_b2(codes, meta, b)
    got = b2.cpu().numpy()
    val = np.where(got == 0x80, 0.0, np.where(got & 8, -1.0, 1.0) * 2.0 ** -(got & 7).astype(np.float64))
    assert np.array_equal(val, ref)


@pytest.mark.parametrize("b", [2, 3, 4])
@pytest.mark.parametrize("g", [8, 16, 32, 64, 128])
def test_geo_quantizer_on_the_midpoints(goq, g, b):
    """Weights on, just above and just below every decision boundary of the lattice (midpoints times the block's largest, which
    is not a power of two), at ordinary, subnormal-threatening and large scales: codes equal to the oracle's."""
    rng = np.random.default_rng(g + b)
    n, k = 24, 2 * g
    emax = (1 << (b - 1)) - 1
    mids = [0.75 * 2.0 ** -e for e in range(emax)] + [2.0 ** -emax, 2.0 ** -(emax + 1)]
    w = np.zeros((n, k), dtype=np.float32)
    for r in range(n):
        top = np.float32(rng.uniform(0.5, 1.0)) * np.float32(2.0 ** [0, -40, -120, 90][r % 4])
        v = (rng.choice(mids, size=k) * np.float64(top)).astype(np.float32)
        step = rng.integers(-1, 2, size=k)
        v = np.where(step > 0, np.nextafter(v, np.float32(np.inf)), np.where(step < 0, np.nextafter(v, np.float32(0)), v))
        w[r] = v * rng.choice(np.array([-1, 1], dtype=np.float32), size=k)
        w[r, ::g] = top * (1 if r % 2 else -1)
    codes_o, _, _ = O.quantize_geo(w, g, b)
    d = goq.desc(n, k, g, b)
    codes = torch.empty((n, k), dtype=torch.uint8, device="cuda")
    meta = torch.empty((n, k // 8), dtype=torch.uint8, device="cuda")
    coef = torch.empty((n, k // g, 2), dtype=torch.int16, device="cuda")
    goq.quantize_geo(d, torch.from_numpy(w).cuda(), codes, meta, coef)
    torch.cuda.synchronize()
    assert np.array_equal(codes.cpu().numpy(), codes_o)


@pytest.mark.parametrize("n,k,g,b,m", [(1, 8, 8, 3, 4), (9, 24, 8, 2, 5), (130, 48, 16, 4, 9), (8, 64, 32, 3, 16), (31, 96, 32, 3, 17),
                                       (200, 192, 64, 3, 32), (7, 128, 64, 2, 33), (300, 256, 128, 3, 64), (129, 384, 128, 3, 65),
                                       (2500, 128, 128, 4, 200)])
def test_ref_solve_edges(goq, n, k, g, b, m):
    """Both sides of the line between the observation form and the Gram form (m = g / 2), row tiles and observation chunks that
    do not fill, every group size. float64 normal equations: 1e-9 as in the general test."""
    w = si.gaussian_weights(n, k, seed=n + m).astype(np.float32)
    codes, meta, _ = O.quantize_geo(w, g, b)
    x = si.f32_activations(m, k, seed=m).astype(np.float32)
    c_ref = O.solve_ref(w, codes, meta, x, g, b, lam=1e-2)
    d = goq.desc(n, k, g, b)
    coef = torch.zeros((n, k // g, 2), dtype=torch.int16, device="cuda")
    c64 = torch.full((n, k // g, 2), np.nan, dtype=torch.float64, device="cuda")
    goq.solve_ref(d, torch.from_numpy(w).cuda(), torch.from_numpy(codes).cuda(), torch.from_numpy(meta).cuda(),
                  torch.from_numpy(x).cuda(), m, 1e-2, coef, c64)
    torch.cuda.synchronize()
    got = c64.cpu().numpy()
    assert np.allclose(got, c_ref, rtol=1e-9, atol=1e-11)
    assert np.array_equal(coef.cpu().numpy().view(np.uint16), got.astype(np.float16).view(np.uint16))


@pytest.mark.parametrize("n,k,g,b,m", [
    (1, 8, 8, 3, 17), (129, 136, 8, 3, 33), (127, 256, 16, 4, 32), (128, 128, 128, 3, 64),
    (4000, 384, 128, 3, 65), (250, 512, 8, 4, 200), (257, 1152, 64, 3, 256), (300, 640, 128, 4, 257), (1000, 4096, 32, 3, 511),
    (130, 8192, 128, 2, 40), (2400, 256, 64, 3, 20), (1100, 2304, 128, 3, 200)])
def test_mid_batch_gemm_edges(goq, n, k, g, b, m):
    """The kernel between decode and prefill: channel tiles and token tiles that do not fill, one unit in all, one tile shared by
    many SMs and several tiles an SM, both operand forms (exact up to 32 tokens), every bit width; twice, bit for bit.
    Bounds: two exact operands with fp32 sums 2e-5 (as every fp32-accumulating kernel), w_hat rounded once to fp16 5e-4."""
    from tests.gpu_util import check_parity, dev, pack_weights
    codes, meta, coef = si.random_quantized(n, k, g, b, seed=n + k + m)
    d, packed = pack_weights(n, k, g, b, codes, meta, coef)
    xb = si.bf16_activations(m, k, seed=m)
    y_ref = O.linear_f64(codes, meta, coef, si.bf16_bits_to_f64(xb), g, b)
    ws = goq.new_workspace(d, goq.OP_GEMM, m)
    prev = goq.set_gemv_variant(4)
    try:
        out = []
        for _ in range(2):
            y = torch.full((m, n), float("nan"), dtype=torch.float32, device="cuda")
            goq.gemm(d, packed, dev(xb), m, goq.BF16, y=y, y_dtype=goq.F32, ws=ws)
            torch.cuda.synchronize()
            assert goq.workspace_status(ws) == goq.OK
            out.append(y.cpu().numpy())
    finally:
        goq.set_gemv_variant(prev)
    assert np.array_equal(out[0], out[1])
    exact = m <= 32
    check_parity(out[0].astype(np.float64), y_ref, 2e-5 if exact else 5e-4, 1e-4 if exact else 2e-3)


@pytest.mark.parametrize("n,k,g,m", [(20000, 128, 128, 64), (20000, 64, 64, 200), (3000, 256, 128, 40), (1024, 2048, 128, 250)])
def test_mid_batch_gemm_back_to_back_on_one_scratch_buffer(goq, n, k, g, m):
    """Calls that follow one another without a wait in between: the second overwrites the fp16 activations and the parked parts of the
    first, and a copy on the same stream reads each output. One k-block (no tile is shared, nothing to add behind the kernel) with
    more units than SMs, and shapes with shared tiles. Every output as from a call of its own, bit for bit."""
    from tests.gpu_util import dev, pack_weights
    codes, meta, coef = si.random_quantized(n, k, g, 3, seed=n + k)
    d, packed = pack_weights(n, k, g, 3, codes, meta, coef)
    ws = goq.new_workspace(d, goq.OP_GEMM, m)
    xs = [dev(si.bf16_activations(m, k, seed=s)) for s in range(4)]
    y = torch.empty((m, n), dtype=torch.float32, device="cuda")
    alone = []
    prev = goq.set_gemv_variant(4)
    try:
        for x in xs:
            goq.gemm(d, packed, x, m, goq.BF16, y=y, y_dtype=goq.F32, ws=ws)
            torch.cuda.synchronize()
            alone.append(y.clone())
        for _ in range(10):
            got = []
            for x in xs:
                goq.gemm(d, packed, x, m, goq.BF16, y=y, y_dtype=goq.F32, ws=ws)
                got.append(y.clone())
            torch.cuda.synchronize()
            assert all(torch.equal(a, c) for a, c in zip(got, alone))
    finally:
        goq.set_gemv_variant(prev)
    assert goq.workspace_status(ws) == goq.OK


@pytest.mark.parametrize("n,k,g,b,m", [(300, 512, 128, 3, 16), (300, 512, 128, 3, 17), (129, 256, 64, 4, 32), (200, 384, 16, 2, 20), (300, 512, 128, 3, 100),
                                       (256, 136, 8, 4, 60), (128, 1024, 128, 3, 700)])
def test_gemm_non_finite_activations_stay_with_their_token(goq, n, k, g, b, m):
    """A token with an infinite element and one with a NaN: every output of theirs is non-finite (an infinity times a weight is one, times
    the zero state NaN); the other tokens' outputs do not change by a bit."""
    from tests.gpu_util import pack_weights, run_gemm_bf16
    codes, meta, coef = si.random_quantized(n, k, g, b, seed=n + k + m)
    d, packed = pack_weights(n, k, g, b, codes, meta, coef)
    xb = si.bf16_activations(m, k, seed=m)
    clean = run_gemm_bf16(d, packed, xb)
    bad = xb.copy()
    bad[1, 5], bad[m - 1, k - 1], bad[m // 2, k // 2] = 0x7F80, 0xFF80, 0x7FC0   # +inf, -inf, NaN
    got = run_gemm_bf16(d, packed, bad)
    hit = sorted({1, m // 2, m - 1})
    rest = [t for t in range(m) if t not in hit]
    assert np.isfinite(clean).all() and not np.isfinite(got[hit]).any()
    assert np.isnan(got[m // 2]).all()
    assert np.array_equal(got[rest], clean[rest])
    yh = run_gemm_bf16(d, packed, bad, goq.BF16)
    assert not np.isfinite(yh[hit]).any() and np.isfinite(yh[rest]).all()


@pytest.mark.parametrize("n,k,g,b,m", [(9472, 256, 64, 3, 200), (9473, 256, 64, 3, 256), (18944, 768, 128, 4, 33), (18945, 256, 128, 3, 100), (9600, 128, 128, 3, 64),
                                       (9600, 1024, 128, 2, 64), (7984, 2048, 128, 3, 20), (8000, 2048, 128, 3, 20), (27200, 96, 32, 4, 32),
                                       (9500, 512, 8, 4, 150), (4096, 1024, 16, 3, 1200), (4096, 1024, 16, 3, 520)])
def test_gemm_either_side_of_the_dispatch_lines(goq, n, k, g, b, m):
    """Automatic dispatch next to its lines (148 SMs): channel tiles that half fill, fill and overfill one wave, one and eight k-blocks; up
    to 32 tokens the units and tiles where the mid-batch kernel takes over from the decode launches; above 256 either estimate.
    Sampled channels of every token: 2e-5 up to 32 tokens, w_hat rounded once to fp16 5e-4 above."""
    from tests.gpu_util import check_parity, pack_weights, run_gemm_bf16
    codes, meta, coef = si.random_quantized(n, k, g, b, seed=n + k + m)
    d, packed = pack_weights(n, k, g, b, codes, meta, coef)
    xb = si.bf16_activations(m, k, seed=m)
    rows = np.unique(np.concatenate([si.sample_rows(n, 200, seed=2), np.arange(n - 20, n)]))
    y_ref = O.linear_f64(codes, meta, coef, si.bf16_bits_to_f64(xb), g, b, rows=rows)
    y = run_gemm_bf16(d, packed, xb)
    assert np.isfinite(y).all()
    check_parity(y[:, rows], y_ref, 2e-5 if m <= 32 else 5e-4, 1e-4 if m <= 32 else 2e-3)


@pytest.mark.parametrize("n,k,g,b", [(200, 384, 16, 3), (130, 136, 8, 3), (257, 512, 8, 4), (64, 1024, 16, 4), (1, 8, 8, 4), (300, 256, 32, 4)])
def test_gemm_up_to_32_rows_is_fp32_accurate_in_every_group(goq, n, k, g, b):
    """Automatic dispatch at 1, 16, 17 and 32 rows, narrow groups and the largest records (W4 in groups of 8: two pieces a copy) among
    them, also in a buffer sized for one row: 2e-5 as for every fp32-accumulating kernel; a single output, which may be small by
    cancellation, within 2^-20 of its terms' magnitudes (fp32 sums of exact products)."""
    from tests.gpu_util import check_parity, dev, pack_weights
    codes, meta, coef = si.random_quantized(n, k, g, b, seed=n + k)
    d, packed = pack_weights(n, k, g, b, codes, meta, coef)
    w = O.decode_b1(codes, b) * np.repeat(coef[..., 0].astype(np.float64), g, 1) + O.decode_b2(codes, meta, b) * np.repeat(coef[..., 1].astype(np.float64), g, 1)
    for m, sized_for in ((1, 1), (16, 16), (17, 17), (32, 32), (32, 1)):
        xb = si.bf16_activations(m, k, seed=m)
        x = si.bf16_bits_to_f64(xb)
        y_ref = O.linear_f64(codes, meta, coef, x, g, b)
        y = torch.full((m, n), float("nan"), dtype=torch.float32, device="cuda")
        try:
            goq.gemm(d, packed, dev(xb), m, goq.BF16, y=y, y_dtype=goq.F32, ws=goq.new_workspace(d, goq.OP_GEMM, sized_for))
        except goq.GoqError as e:   # less scratch than documented may be refused
            assert sized_for < m and e.status == goq.ERR_WORKSPACE
            continue
        torch.cuda.synchronize()
        got = y.cpu().numpy().astype(np.float64)
        if n > 1:
            check_parity(got, y_ref, 2e-5, 1e-4)
        else:
            assert (np.abs(got - y_ref) <= 2.0 ** -20 * np.abs(x) @ np.abs(w).T).all()


@pytest.mark.parametrize("n,k,g,b,largest,ms", [(4096, 4096, 128, 3, 257, (17, 100, 256)), (1024, 2048, 16, 3, 300, (20, 32, 200, 256)),
                                                (2048, 1024, 64, 4, 2048, (18, 33, 255, 700))])
def test_gemm_on_a_buffer_for_a_larger_batch(goq, n, k, g, b, largest, ms):
    """A scratch buffer sized for a larger batch: the same kernel, so the same bits, as with a buffer of the call's own size."""
    from tests.gpu_util import dev, pack_weights, run_gemm_bf16
    codes, meta, coef = si.random_quantized(n, k, g, b, seed=n + k)
    d, packed = pack_weights(n, k, g, b, codes, meta, coef)
    ws = goq.new_workspace(d, goq.OP_GEMM, largest)
    for m in ms:
        xb = si.bf16_activations(m, k, seed=m)
        y = torch.full((m, n), float("nan"), dtype=torch.float32, device="cuda")
        goq.gemm(d, packed, dev(xb), m, goq.BF16, y=y, y_dtype=goq.F32, ws=ws)
        torch.cuda.synchronize()
        assert np.array_equal(y.cpu().numpy().astype(np.float64), run_gemm_bf16(d, packed, xb))


@pytest.mark.parametrize("n,k,g,b,m", [(4000, 8192, 128, 3, 200), (4000, 8192, 128, 3, 20)])
def test_mid_batch_gemm_reports_a_wait_that_runs_out(goq, n, k, g, b, m):
    """With one poll for the accumulator the mid-batch kernel gives up, either operand form: the status word reads GOQ_ERR_TIMEOUT, the
    context stays usable, and on a fresh scratch buffer the next call is right again."""
    from tests.gpu_util import dev, pack_weights
    codes, meta, coef = si.random_quantized(n, k, g, b, seed=n + k)
    d, packed = pack_weights(n, k, g, b, codes, meta, coef)
    x = dev(si.bf16_activations(m, k, seed=m))
    ws = goq.new_workspace(d, goq.OP_GEMM, m)

    def call():
        y = torch.zeros((m, n), dtype=torch.float32, device="cuda")
        goq.gemm(d, packed, x, m, goq.BF16, y=y, y_dtype=goq.F32, ws=ws)
        torch.cuda.synchronize()
        return y, goq.workspace_status(ws)
    prev = goq.set_gemv_variant(4)
    try:
        good, status = call()
        assert status == goq.OK
        goq.set_wait_limit(1)
        assert call()[1] == goq.ERR_TIMEOUT
        goq.set_wait_limit(0)
        goq.workspace_init(ws)
        again, status = call()
        assert status == goq.OK and torch.equal(good, again)
    finally:
        goq.set_wait_limit(0)
        goq.set_gemv_variant(prev)


@pytest.mark.parametrize("n,k,g,b,m", [
    (1, 32, 32, 3, 1), (129, 160, 32, 4, 33), (127, 256, 64, 2, 48), (128, 128, 128, 3, 16), (4000, 384, 128, 3, 17), (300, 640, 128, 4, 64),
    (1000, 4096, 32, 3, 65), (130, 8192, 128, 2, 40), (2400, 256, 64, 3, 128), (19200, 128, 128, 3, 24), (257, 1152, 64, 4, 129), (1100, 2304, 128, 3, 200)])
def test_e4m3_operand_gemm_edges(goq, n, k, g, b, m):
    """Both bases and the activations as e4m3 numbers: channel and token tiles that do not fill, every bit width and number of macro-blocks a
    k-block, one unit in all, one tile shared by many SMs, tiles an SM has whole; tokens of tiny and huge magnitude, of zeros, and with one element 2^14
    times the others (what such an element leaves of the others: the next test but one). Twice, bit for bit, two calls back to back. Bounds as for every
    fp32-accumulating kernel."""
    from tests.gpu_util import check_parity, dev, pack_weights
    codes, meta, coef = si.random_quantized(n, k, g, b, seed=n + k + m)
    d, packed = pack_weights(n, k, g, b, codes, meta, coef)
    x = si.bf16_bits_to_f64(si.bf16_activations(m, k, seed=m))
    x[0, k // 2] *= 2.0 ** 14
    if m > 3:
        x[1] *= 2.0 ** -100
        x[2] *= 2.0 ** 100
        x[3] = 0.0
    xb = si.f32_to_bf16_bits(x.astype(np.float32))
    y_ref = O.linear_f64(codes, meta, coef, si.bf16_bits_to_f64(xb), g, b)
    ws = goq.new_workspace(d, goq.OP_GEMM, m)
    prev = goq.set_gemv_variant(6)
    try:
        out = [torch.full((m, n), float("nan"), dtype=torch.float32, device="cuda") for _ in range(2)]
        y16 = torch.full((m, n), float("nan"), dtype=torch.bfloat16, device="cuda")
        for y in out:
            goq.gemm(d, packed, dev(xb), m, goq.BF16, y=y, y_dtype=goq.F32, ws=ws)
        goq.gemm(d, packed, dev(xb), m, goq.BF16, y=y16, y_dtype=goq.BF16, ws=ws)
        torch.cuda.synchronize()
        assert goq.workspace_status(ws) == goq.OK
    finally:
        goq.set_gemv_variant(prev)
    assert torch.equal(out[0], out[1]) and torch.equal(y16, out[0].to(torch.bfloat16))
    got = out[0].cpu().numpy().astype(np.float64)
    scale = np.ones((m, 1))
    if m > 3:
        scale[1], scale[2] = 2.0 ** 100, 2.0 ** -100   # tokens of one magnitude again, for the element-wise bound
        assert not got[3].any()
    check_parity(got * scale, y_ref * scale, 2e-5, 1e-4)


@pytest.mark.parametrize("n,k,g,b,m", [(8192, 4096, 128, 4, 4), (12000, 4096, 128, 3, 16), (9000, 8192, 64, 2, 9), (4000, 4096, 128, 3, 30), (16000, 512, 64, 4, 17),
                                       (4096, 4096, 64, 3, 64), (2048, 2048, 128, 3, 128), (8192, 2048, 128, 3, 128)])
def test_calls_either_side_of_the_lines_of_the_e4m3_kernel(goq, n, k, g, b, m):
    """Automatic dispatch next to the lines of that kernel, through goq_gemm and (up to 16 tokens) goq_gemv, with a buffer of the documented size and, for
    goq_gemv at W4, with none. Sampled channels; 2e-5 up to 32 tokens, 5e-4 (w_hat rounded once to fp16) above."""
    from tests.gpu_util import check_parity, dev, pack_weights, run_gemm_bf16, run_gemv
    codes, meta, coef = si.random_quantized(n, k, g, b, seed=n + k + m)
    d, packed = pack_weights(n, k, g, b, codes, meta, coef)
    xb = si.bf16_activations(m, k, seed=m)
    rows = np.unique(np.concatenate([si.sample_rows(n, 200, seed=2), np.arange(n - 20, n)]))
    y_ref = O.linear_f64(codes, meta, coef, si.bf16_bits_to_f64(xb), g, b, rows=rows)
    tol = (2e-5, 1e-4) if m <= 32 else (5e-4, 2e-3)
    check_parity(run_gemm_bf16(d, packed, xb)[:, rows], y_ref, *tol)
    if m <= 16:
        check_parity(run_gemv(d, packed, xb)[:, rows], y_ref, *tol)
        if b == 4:
            y = torch.full((m, n), float("nan"), dtype=torch.float32, device="cuda")
            goq.gemv(d, packed, dev(xb), m, y, goq.F32)
            torch.cuda.synchronize()
            check_parity(y.cpu().numpy().astype(np.float64)[:, rows], y_ref, *tol)


@pytest.mark.parametrize("n,k,g,b,m,variant", [(16384, 4096, 128, 4, 4, 0), (12000, 4096, 128, 3, 16, 0), (28672, 2048, 64, 2, 11, 0), (300, 640, 32, 3, 24, 6), (130, 128, 128, 2, 40, 6),
                                               (8192, 4096, 128, 3, 32, 0)])
def test_small_elements_beside_a_large_one_and_non_finite_ones_in_e4m3_operands(goq, n, k, g, b, m, variant):
    """One element of a token 2^13 .. 2^40 times the others, and channels whose states are zero there: to them the token is an ordinary one, and their
    outputs are held to their own magnitude, by the bounds of every fp32-accumulating kernel. An infinite or NaN element gives what Eq. 4 gives: infinite or
    NaN channel by channel. Through goq_gemm and (up to 16 tokens) goq_gemv; every other token is that of a call without these elements, bit for bit."""
    from tests.gpu_util import check_parity, pack_weights, run_gemm_bf16, run_gemv
    codes, meta, coef = si.random_quantized(n, k, g, b, seed=n + k + m)
    at, blind = k // 2 + 3, np.arange(0, n, 3)   # channels that do not see the micro-block of that element
    mb = at // 8 * 8
    codes[blind, mb:mb + 8] = (1 << (b - 1)) - 1
    d, packed = pack_weights(n, k, g, b, codes, meta, coef)
    plain = si.bf16_activations(m, k, seed=m)
    x = si.bf16_bits_to_f64(plain)
    powers = [2.0 ** e for e in (13, 16, 22, 28, 40)][:m - 2]
    for tok, f in enumerate(powers):
        x[tok, at] = f * 1.5
    xb = si.f32_to_bf16_bits(x.astype(np.float32))
    xb[m - 2, at] = 0x7F80 if m % 2 else 0xFF80
    xb[m - 1, at] = 0x7FC0
    rows = np.unique(np.concatenate([blind[si.sample_rows(len(blind), min(len(blind), 150), seed=2)], si.sample_rows(n, min(n, 150), seed=3), np.arange(n - 20, n)]))
    with np.errstate(invalid="ignore"):
        y_ref = O.linear_f64(codes, meta, coef, si.bf16_bits_to_f64(xb), g, b, rows=rows)
    unseen = np.isin(rows, blind)
    for run in (run_gemm_bf16, run_gemv)[:2 if m <= 16 and variant == 0 else 1]:
        all_y, base = run(d, packed, xb, variant=variant), run(d, packed, plain, variant=variant)
        y = all_y[:, rows]
        for tok in range(len(powers)):
            check_parity(y[tok, unseen], y_ref[tok, unseen], 2e-5, 1e-4, "2^%g" % np.log2(powers[tok]))
        check_parity(y[:m - 2], y_ref[:m - 2], 2e-5, 1e-4)
        for tok in (m - 2, m - 1):
            assert np.array_equal(np.isnan(y[tok]), np.isnan(y_ref[tok])) and np.array_equal(np.isposinf(y[tok]), np.isposinf(y_ref[tok]))
            assert np.array_equal(np.isneginf(y[tok]), np.isneginf(y_ref[tok]))
        assert np.array_equal(all_y[len(powers):m - 2], base[len(powers):m - 2])


@pytest.mark.parametrize("variant,n,k,g,b,m", [(0, 144, 512, 64, 3, 200), (4, 300, 640, 16, 4, 70), (3, 260, 512, 128, 3, 400), (3, 130, 256, 8, 2, 300)])
def test_small_elements_beside_a_large_one_in_fp16_operands(goq, variant, n, k, g, b, m):
    """The kernels with an fp16 copy of the activations: one element of a token 2^13 .. 2^24 times the others, channels whose states are zero there, held to
    their own magnitude. fp16 holds 2^-28 of a token's largest element with bf16's eight bits; w_hat rounded once: 5e-4."""
    from tests.gpu_util import check_parity, pack_weights, run_gemm_bf16
    codes, meta, coef = si.random_quantized(n, k, g, b, seed=n + k + m)
    at, blind = k // 2 + 3, np.arange(0, n, 3)
    mb = at // 8 * 8
    codes[blind, mb:mb + 8] = (1 << (b - 1)) - 1
    d, packed = pack_weights(n, k, g, b, codes, meta, coef)
    x = si.bf16_bits_to_f64(si.bf16_activations(m, k, seed=m))
    powers = (13, 16, 20, 24)
    for tok, e in enumerate(powers):
        x[tok, at] = 1.5 * 2.0 ** e
    xb = si.f32_to_bf16_bits(x.astype(np.float32))
    y_ref = O.linear_f64(codes, meta, coef, si.bf16_bits_to_f64(xb), g, b)
    y = run_gemm_bf16(d, packed, xb, variant=variant)
    for tok, e in enumerate(powers):
        check_parity(y[tok, blind], y_ref[tok, blind], 5e-4, 2e-3, "2^%d" % e)
    check_parity(y, y_ref, 5e-4, 2e-3)


@pytest.mark.parametrize("n,k,g,m", [(16384, 4096, 128, 4), (9000, 8192, 128, 16)])
def test_tokens_that_e4m3_operands_do_not_hold_are_the_fragment_kernels(goq, n, k, g, m):
    """W4: a token whose elements span 2^28 is computed from its bf16 elements, bit for bit as goq_gemv without scratch (the fragment kernel) has it; one with
    a few tiny elements among ordinary ones keeps to its slices (within fp32 sums of the other, not the same bits)."""
    from tests.gpu_util import dev, pack_weights, run_gemv
    codes, meta, coef = si.random_quantized(n, k, g, 4, seed=n + k)
    d, packed = pack_weights(n, k, g, 4, codes, meta, coef)
    x = si.bf16_bits_to_f64(si.bf16_activations(m, k, seed=m))
    x[1, 5] = 2.0 ** 28
    x[2, 7:10] = 1e-12
    xb = si.f32_to_bf16_bits(x.astype(np.float32))
    y = run_gemv(d, packed, xb)
    y0 = torch.zeros((m, n), dtype=torch.float32, device="cuda")
    goq.gemv(d, packed, dev(xb), m, y0, goq.F32)
    torch.cuda.synchronize()
    y0 = y0.cpu().numpy().astype(np.float64)
    assert np.array_equal(y[1], y0[1])
    for tok in (0, 2, m - 1):
        assert 0 < np.linalg.norm(y[tok] - y0[tok]) <= 1e-6 * np.linalg.norm(y0[tok]), tok


def test_e4m3_operand_gemm_reports_a_wait_that_runs_out(goq):
    """With one poll a wait the kernel gives up: the status word reads GOQ_ERR_TIMEOUT, and on a fresh scratch buffer the next call is right again."""
    from tests.gpu_util import dev, pack_weights
    n, k, g, b, m = 4000, 8192, 128, 3, 40
    codes, meta, coef = si.random_quantized(n, k, g, b, seed=n + k)
    d, packed = pack_weights(n, k, g, b, codes, meta, coef)
    x = dev(si.bf16_activations(m, k, seed=m))
    ws = goq.new_workspace(d, goq.OP_GEMM, m)

    def call():
        y = torch.zeros((m, n), dtype=torch.float32, device="cuda")
        goq.gemm(d, packed, x, m, goq.BF16, y=y, y_dtype=goq.F32, ws=ws)
        torch.cuda.synchronize()
        return y, goq.workspace_status(ws)
    prev = goq.set_gemv_variant(6)
    try:
        good, status = call()
        assert status == goq.OK
        goq.set_wait_limit(1)
        assert call()[1] == goq.ERR_TIMEOUT
        goq.set_wait_limit(0)
        goq.workspace_init(ws)
        again, status = call()
        assert status == goq.OK and torch.equal(good, again)
    finally:
        goq.set_wait_limit(0)
        goq.set_gemv_variant(prev)


@pytest.mark.parametrize("n,k,g,b,m", [
    (40, 64, 32, 3, 257),        # one channel tile: the pair's second CTA has none; one k-block, half of it padding
    (300, 640, 64, 4, 300),      # three tiles, W4
    (260, 256, 16, 2, 1000),     # token tiles that do not fill, narrow groups
    (19000, 128, 128, 3, 513),   # one more pair of tiles than pairs of SMs: the last ones as token halves
    (9600, 512, 128, 3, 600),    # full and half tiles in one launch
    (512, 2176, 128, 2, 4100),
    (4096, 4096, 128, 3, 2048)])  # every pair busy: records, stages and hops at full rate
def test_prefill_gemm_on_pairs_of_sms_edges(goq, n, k, g, b, m):
    """More than 256 tokens: channel tiles, token tiles and k that do not fill a pair, twice back to back, bit for bit. w_hat rounded once to fp16: 5e-4."""
    from tests.gpu_util import check_parity, dev, pack_weights
    codes, meta, coef = si.random_quantized(n, k, g, b, seed=n + k + m)
    d, packed = pack_weights(n, k, g, b, codes, meta, coef)
    xb = si.bf16_activations(m, k, seed=m)
    rows = np.unique(np.concatenate([si.sample_rows(n, min(n, 150), seed=2), np.arange(n - 20, n)]))
    y_ref = O.linear_f64(codes, meta, coef, si.bf16_bits_to_f64(xb), g, b, rows=rows)
    ws = goq.new_workspace(d, goq.OP_GEMM, m)
    out = [torch.full((m, n), float("nan"), dtype=torch.float32, device="cuda") for _ in range(2)]
    y16 = torch.full((m, n), float("nan"), dtype=torch.bfloat16, device="cuda")
    prev = goq.set_gemv_variant(3)   # the prefill kernels whatever the estimates
    try:
        for y in out:
            goq.gemm(d, packed, dev(xb), m, goq.BF16, y=y, y_dtype=goq.F32, ws=ws)
        goq.gemm(d, packed, dev(xb), m, goq.BF16, y=y16, y_dtype=goq.BF16, ws=ws)
        torch.cuda.synchronize()
    finally:
        goq.set_gemv_variant(prev)
    assert goq.workspace_status(ws) == goq.OK
    assert torch.equal(out[0], out[1]) and torch.equal(y16, out[0].to(torch.bfloat16))
    check_parity(out[0].cpu().numpy().astype(np.float64)[:, rows], y_ref, 5e-4, 2e-3)


def test_prefill_gemm_on_pairs_of_sms_reads_no_tile_of_the_call_before(goq):
    """Every pair busy, two sets of weights and activations in turn on one scratch buffer: a weight tile that an MMA read before the other CTA's part of it was in
    place would carry the other call's weights. Every call repeats its first result bit for bit."""
    from tests.gpu_util import check_parity, dev, pack_weights
    n, k, g, b, m = 4096, 2048, 128, 3, 1536
    calls, rows = [], si.sample_rows(n, 100, seed=2)
    for seed in (1, 2):
        codes, meta, coef = si.random_quantized(n, k, g, b, seed=seed)
        d, packed = pack_weights(n, k, g, b, codes, meta, coef)
        xb = si.bf16_activations(m, k, seed=seed)
        calls.append((d, packed, dev(xb), O.linear_f64(codes, meta, coef, si.bf16_bits_to_f64(xb), g, b, rows=rows)))
    ws = goq.new_workspace(calls[0][0], goq.OP_GEMM, m)
    prev = goq.set_gemv_variant(3)
    try:
        out = [torch.zeros((m, n), dtype=torch.float32, device="cuda") for _ in range(24)]
        for i, y in enumerate(out):
            d, packed, x, _ = calls[i % 2]
            goq.gemm(d, packed, x, m, goq.BF16, y=y, y_dtype=goq.F32, ws=ws)
        torch.cuda.synchronize()
    finally:
        goq.set_gemv_variant(prev)
    assert goq.workspace_status(ws) == goq.OK
    for i, y in enumerate(out):
        assert torch.equal(y, out[i % 2]), i
    for i in range(2):
        check_parity(out[i].cpu().numpy().astype(np.float64)[:, rows], calls[i][3], 5e-4, 2e-3)


@pytest.mark.parametrize("n,k,g,b,m", [(4000, 2048, 128, 3, 600), (300, 128, 64, 4, 300)])   # many chunks; as many as there are stages or fewer
def test_prefill_gemm_on_pairs_of_sms_reports_a_wait_that_runs_out(goq, n, k, g, b, m):
    """With one poll a wait either CTA of a pair gives up by itself and both end: the status word reads GOQ_ERR_TIMEOUT, and on a fresh scratch buffer the next
    call is right again."""
    from tests.gpu_util import dev, pack_weights
    codes, meta, coef = si.random_quantized(n, k, g, b, seed=n + k)
    d, packed = pack_weights(n, k, g, b, codes, meta, coef)
    x = dev(si.bf16_activations(m, k, seed=m))
    ws = goq.new_workspace(d, goq.OP_GEMM, m)

    def call():
        y = torch.zeros((m, n), dtype=torch.float32, device="cuda")
        goq.gemm(d, packed, x, m, goq.BF16, y=y, y_dtype=goq.F32, ws=ws)
        torch.cuda.synchronize()
        return y, goq.workspace_status(ws)
    prev = goq.set_gemv_variant(3)
    try:
        good, status = call()
        assert status == goq.OK
        goq.set_wait_limit(1)
        assert call()[1] == goq.ERR_TIMEOUT
        goq.set_wait_limit(0)
        goq.workspace_init(ws)
        again, status = call()
        assert status == goq.OK and torch.equal(good, again)
    finally:
        goq.set_wait_limit(0)
        goq.set_gemv_variant(prev)


@pytest.mark.parametrize("variant,n,k,g,b,m", [
    (3, 1, 8, 8, 3, 257), (3, 130, 256, 64, 2, 513), (3, 33, 136, 8, 3, 600), (3, 384, 384, 32, 4, 1025), (3, 9600, 128, 128, 3, 1024),
    (3, 9500, 64, 64, 3, 1030), (4, 20000, 256, 128, 3, 300), (4, 5000, 128, 32, 4, 1025), (0, 4100, 256, 64, 3, 700)])
def test_prefill_gemm_token_tiles(goq, variant, n, k, g, b, m):
    """Equal token tiles narrower than 512: one token more than a half tile holds, a last tile that does not fill, tiles left over
    as halves (9600 and 9500 channels on 148 SMs), few channel tiles in many token tiles; in the mid-batch kernel ranges of several
    whole tiles, drained by four warps. Every token's row is written once. Bound: w_hat rounded once to fp16, 5e-4."""
    from tests.gpu_util import check_parity, dev, pack_weights
    codes, meta, coef = si.random_quantized(n, k, g, b, seed=n + k + m)
    d, packed = pack_weights(n, k, g, b, codes, meta, coef)
    xb = si.bf16_activations(m, k, seed=m)
    y_ref = O.linear_f64(codes, meta, coef, si.bf16_bits_to_f64(xb), g, b)
    ws = goq.new_workspace(d, goq.OP_GEMM, m)
    prev = goq.set_gemv_variant(variant)
    try:
        y = torch.full((m, n), float("nan"), dtype=torch.float32, device="cuda")
        goq.gemm(d, packed, dev(xb), m, goq.BF16, y=y, y_dtype=goq.F32, ws=ws)
        torch.cuda.synchronize()
        assert goq.workspace_status(ws) == goq.OK
    finally:
        goq.set_gemv_variant(prev)
    got = y.cpu().numpy().astype(np.float64)
    if n > 1:
        check_parity(got, y_ref, 5e-4, 2e-3)
    else:
        # One output has no norm over channels to average in, and it may be small by cancellation. Each w_hat is off by at most its
        # fp16 rounding, 2^-11 of itself (the sums in fp32 add far less), so the output by at most 2^-11 sum |x| |w_hat|.
        w = np.abs(O.decode_b1(codes, b) * np.repeat(coef[..., 0].astype(np.float64), g, 1)
                   + O.decode_b2(codes, meta, b) * np.repeat(coef[..., 1].astype(np.float64), g, 1))
        assert (np.abs(got - y_ref) <= 2.0 ** -11 * np.abs(si.bf16_bits_to_f64(xb)) @ w.T).all()


@pytest.mark.parametrize("n,k,g,b,m", [(1, 32, 32, 3, 1), (16, 128, 128, 2, 4), (2368, 128, 128, 3, 3), (2369, 128, 64, 3, 1), (37888, 256, 32, 2, 2),
                                       (16, 12288, 128, 3, 4), (129, 3200, 64, 3, 3), (4736, 4096, 128, 3, 1)])
def test_single_decode_gemv_edges(goq, n, k, g, b, m):
    """The single-linear integer-operand kernel: one record in all, one record an SM, a tile spread over all SMs, several tiles an SM,
    ranges that need all or few of the k-blocks; back to back on one scratch buffer, whose counter area must stay zero, and equal
    to the same linear in a chain bit for bit. Bound 2e-5 as for every fp32-accumulating kernel."""
    from tests.gpu_util import check_parity, dev, pack_weights
    codes, meta, coef = si.random_quantized(n, k, g, b, seed=n + k + m)
    d, packed = pack_weights(n, k, g, b, codes, meta, coef)
    xs = [si.bf16_activations(m, k, seed=s) for s in range(3)]
    ws = goq.new_workspace(d, goq.OP_GEMV, m)
    ys = [torch.full((m, n), float("nan"), dtype=torch.float32, device="cuda") for _ in xs]
    xd = [dev(x) for x in xs]
    prev = goq.set_gemv_variant(5)
    try:
        for x, y in zip(xd, ys):
            goq.gemv(d, packed, x, m, y, goq.F32, ws=ws)
    finally:
        goq.set_gemv_variant(prev)
    torch.cuda.synchronize()
    assert goq.workspace_status(ws) == goq.OK and not ws[256:256 + 65536].any()
    rows = si.sample_rows(n, min(n, 200), seed=1)
    for x, y in zip(xs, ys):
        y_ref = O.linear_f64(codes, meta, coef, si.bf16_bits_to_f64(x), g, b, rows=rows)
        got = y.cpu().numpy().astype(np.float64)[:, rows]
        if n > 1:
            check_parity(got, y_ref, 2e-5, 1e-4)
        else:
            # One output has no norm over channels to average in, and it may be small by cancellation. An activation is rounded at
            # half of 2^-14 of the largest of its block, so the output is off by at most 2^-15 max|x| sum |w_hat|.
            w = np.abs(O.decode_b1(codes, b) * np.repeat(coef[..., 0].astype(np.float64), g, 1)
                       + O.decode_b2(codes, meta, b) * np.repeat(coef[..., 1].astype(np.float64), g, 1)).sum()
            assert np.abs(got - y_ref).max() <= 2.0 ** -15 * np.abs(si.bf16_bits_to_f64(x)).max() * w
    seq_ws = torch.zeros(goq.sequence_workspace_bytes(1), dtype=torch.uint8, device="cuda")
    yc = torch.empty((m, n), dtype=torch.float32, device="cuda")
    goq.gemv_sequence(goq.make_sequence([(d, packed, xd[0], m, yc, goq.F32, False)]), seq_ws)
    torch.cuda.synchronize()
    assert torch.equal(yc, ys[0])


@pytest.mark.parametrize("b", [2, 3, 4])
@pytest.mark.parametrize("n,k,g,m", [(1, 32, 32, 1), (17, 160, 32, 8), (256, 256, 64, 9), (40, 640, 128, 5), (33, 896, 128, 16), (16, 16384, 128, 16),
                                     (600, 4096, 64, 3), (1200, 2080, 32, 12), (2400, 2048, 128, 7)])
def test_fragment_gemv_edges(goq, n, k, g, m, b):
    """The decode GEMV on bf16 fragments: rows and columns that end inside a record, fewer k-blocks than warps, one CTA per tile and
    clusters of two to eight, odd batches; fp32 and bf16 outputs, twice, bit for bit. fp32 sums of exact products: 2e-5."""
    from tests.gpu_util import check_bf16_output, check_parity, pack_weights, run_gemv
    codes, meta, coef = si.random_quantized(n, k, g, b, seed=n + k + m + b)
    d, packed = pack_weights(n, k, g, b, codes, meta, coef)
    xb = si.bf16_activations(m, k, seed=m)
    y_ref = O.linear_f64(codes, meta, coef, si.bf16_bits_to_f64(xb), g, b)
    y = run_gemv(d, packed, xb, goq.F32)
    check_parity(y, y_ref, 2e-5, 1e-4)
    assert np.array_equal(y, run_gemv(d, packed, xb, goq.F32))
    check_bf16_output(run_gemv(d, packed, xb, goq.BF16), y_ref, 1e-4)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("m,k,abits", [(1, 1, 8), (9, 4, 8), (3, 1024, 8), (17, 1028, 8), (2, 5000, 4), (5, 4096, 2), (3, 4100, 6), (4, 771, 8)])
def test_activation_quantizer_edges(goq, m, k, abits, dtype):
    """Rows of every path (a warp, a CTA, more than the registers hold, not a multiple of four), quotients on and next to the halves
    where the fp32 estimate cannot decide, the largest and smallest scales: integers and scales equal to the oracle's."""
    rng = np.random.default_rng(m * k + abits)
    qmax = 2 ** (abits - 1) - 1
    x = rng.standard_normal((m, k)).astype(np.float32)
    for r in range(m):
        top = np.float32([3.0, 1.7e-30, 2.9e38, 1e-39, 0.3333][r % 5])
        half = (rng.integers(0, 2 * qmax, size=k) - qmax + 0.5) * (np.float64(top) / qmax)
        half = half.astype(np.float32)
        step = rng.integers(-2, 3, size=k)
        half = np.where(step > 0, np.nextafter(half, np.float32(np.inf)), np.where(step < 0, np.nextafter(half, np.float32(-np.inf)), half))
        x[r] = np.clip(np.where(rng.random(k) < 0.7, half, x[r] * top / 5), -top, top)
        x[r, r % k] = top
    if dtype == "bf16":
        bits = si.f32_to_bf16_bits(x)
        x = si.bf16_bits_to_f64(bits).astype(np.float32)
        xd, code = torch.from_numpy(bits.view(np.int16)).cuda(), goq.BF16
    else:
        xd, code = torch.from_numpy(x).cuda(), goq.F32
    xq_ref, sx_ref = O.quantize_activations_int(x, abits)
    for amax in (None, torch.from_numpy(np.abs(x).max(axis=1)).cuda()):
        xq = torch.full((m, k), 99, dtype=torch.int8, device="cuda")
        sx = torch.zeros(m, dtype=torch.float32, device="cuda")
        goq.quantize_activations(xd, code, m, k, xq, sx, amax=amax, abits=abits)
        torch.cuda.synchronize()
        assert np.array_equal(xq.cpu().numpy(), xq_ref)
        assert np.array_equal(sx.cpu().numpy(), sx_ref)


@pytest.mark.parametrize("n,k,g,b,m", [(1, 32, 32, 3, 1), (16, 32, 32, 2, 127), (63, 96, 32, 4, 128), (64, 128, 64, 3, 129), (65, 192, 64, 4, 255),
                                       (130, 320, 64, 2, 256), (200, 1024, 128, 3, 257), (72, 416, 32, 3, 300), (8, 1024, 128, 4, 700),
                                       (4800, 128, 64, 3, 600), (192, 3072, 64, 3, 40000 // 64), (640, 3072, 32, 3, 4200), (192, 768, 32, 2, 1500)])
@pytest.mark.parametrize("out", ["f32", "bf16"])
def test_int8_tensor_core_gemm_edges(goq, n, k, g, b, m, out):
    """The int8 layer on the tensor cores: channel and token tiles that do not fill, one and two token halves a tile, fewer and more tiles
    than SMs, every bit width and group, many rounds of the record ring with the largest records, coefficients over the whole byte (-128 and 0 among them): accumulators bit-exact, outputs
    those accumulators give in fp32 (2^-22 of the two terms' magnitudes), bf16 within its rounding."""
    from tests.gpu_util import dev, pack_weights
    rng = np.random.default_rng(n + k + m)
    codes, meta, coef = si.random_quantized(n, k, g, b, seed=n + k)
    d, packed = pack_weights(n, k, g, b, codes, meta, coef)
    cq = rng.integers(-128, 128, size=(n, k // g, 2)).astype(np.int8)
    cq[0, 0] = (-128, 0)
    x = rng.integers(-127, 128, size=(m, k)).astype(np.int8)
    x[m // 2] = 127
    sx = rng.uniform(0.5, 2, size=m).astype(np.float32)
    sc = rng.uniform(-1, 1, size=(n, 2)).astype(np.float32)
    y = torch.zeros((m, n), dtype=torch.float32 if out == "f32" else torch.bfloat16, device="cuda")
    acc = torch.zeros((2, m, n), dtype=torch.int32, device="cuda")
    goq.gemm(d, packed, dev(x), m, goq.I8, y=y, y_dtype=goq.F32 if out == "f32" else goq.BF16, sx=dev(sx), cq=dev(cq), sc=dev(sc), acc=acc)
    torch.cuda.synchronize()
    rows = si.sample_rows(n, min(n, 256), seed=1)
    a1, a2, _ = O.linear_i32(codes[rows], meta[rows], cq[rows], sc[rows], x, sx, g, b)
    got = acc.cpu().numpy()
    assert np.array_equal(got[0][:, rows], a1) and np.array_equal(got[1][:, rows], a2)
    emax = (1 << (b - 1)) - 1
    t = [sx[:, None].astype(np.float64) * 2.0 ** -emax * sc[rows, i].astype(np.float64) * a for i, a in enumerate((a1, a2))]
    yh = y.float().cpu().numpy().astype(np.float64)[:, rows]
    bound = 2.0 ** -21 * (np.abs(t[0]) + np.abs(t[1])) + (0.0 if out == "f32" else 2.0 ** -8 * np.abs(t[0] + t[1]))
    assert np.all(np.abs(yh - t[0] - t[1]) <= bound)


@pytest.mark.parametrize("n,k,g,b,m", [(65, 192, 64, 3, 129), (64, 128, 32, 4, 5), (40, 64, 16, 2, 33)])
def test_int8_layer_takes_scales_at_any_float_address(goq, n, k, g, b, m):
    """Scale and output arrays that begin one float behind an aligned address, as slices of larger arrays do: same accumulators and
    outputs as at an aligned one, from goq_gemm and from the requantising entry point."""
    from tests.gpu_util import dev, pack_weights
    rng = np.random.default_rng(n)
    codes, meta, coef = si.random_quantized(n, k, g, b, seed=n + k)
    d, packed = pack_weights(n, k, g, b, codes, meta, coef)
    cq = dev(rng.integers(-127, 128, size=(n, k // g, 2)).astype(np.int8))
    x = dev(rng.integers(-127, 128, size=(m, k)).astype(np.int8))
    sx, sc = rng.uniform(0.5, 2, size=m).astype(np.float32), rng.uniform(-1, 1, size=(n, 2)).astype(np.float32)
    got = []
    for shift in (0, 1):
        zeros = np.zeros((m, n), dtype=np.float32)
        y, h = _unaligned(zeros, shift), _unaligned(zeros, shift)
        acc = _unaligned(np.zeros((2, m, n), dtype=np.int32), shift)
        amax, sy = _unaligned(np.zeros(m, dtype=np.float32), shift), _unaligned(np.zeros(m, dtype=np.float32), shift)
        yq = _unaligned(np.zeros((m, n), dtype=np.int8), shift)
        sxd, scd = _unaligned(sx, shift), _unaligned(sc, shift)
        goq.gemm(d, packed, x, m, goq.I8, y=y, y_dtype=goq.F32, sx=sxd, cq=cq, sc=scd, acc=acc)
        goq.gemm_i8_requant(d, packed, x, m, sxd, cq, scd, h, amax, yq, sy)
        torch.cuda.synchronize()
        got.append([t.cpu().numpy().copy() for t in (y, acc, h, amax, yq, sy)])
    assert got[0][1].any() and all(np.array_equal(a, c) for a, c in zip(*got))


def test_int8_layer_reports_a_wait_that_runs_out(goq):
    """With one poll a wait the epilogue of 128 k-blocks runs out of it: the status word of goq_gemm reads GOQ_ERR_TIMEOUT, and the
    requantising entry point, which has no scratch, returns NaN magnitudes and scales. The next calls are right again."""
    from tests.gpu_util import dev, pack_weights
    rng = np.random.default_rng(1)
    n, k, g, b, m = 256, 16384, 128, 3, 300
    codes, meta, coef = si.random_quantized(n, k, g, b, seed=1)
    d, packed = pack_weights(n, k, g, b, codes, meta, coef)
    cq = dev(rng.integers(-127, 128, size=(n, k // g, 2)).astype(np.int8))
    x = dev(rng.integers(-127, 128, size=(m, k)).astype(np.int8))
    sx, sc = torch.rand(m, device="cuda") + 0.5, torch.rand((n, 2), device="cuda") + 0.1
    ws = torch.zeros(1024, dtype=torch.uint8, device="cuda")

    def call():
        y, h = torch.zeros((m, n), device="cuda"), torch.zeros((m, n), device="cuda")
        amax, sy, yq = torch.zeros(m, device="cuda"), torch.zeros(m, device="cuda"), torch.zeros((m, n), dtype=torch.int8, device="cuda")
        goq.gemm(d, packed, x, m, goq.I8, y=y, y_dtype=goq.F32, sx=sx, cq=cq, sc=sc, ws=ws)
        goq.gemm_i8_requant(d, packed, x, m, sx, cq, sc, h, amax, yq, sy)
        torch.cuda.synchronize()
        return y, h, amax, sy, yq
    good = call()
    assert goq.workspace_status(ws) == goq.OK and torch.isfinite(good[2]).all() and torch.equal(good[0], good[1])
    goq.set_wait_limit(1)
    try:
        cut = call()
    finally:
        goq.set_wait_limit(0)
    assert goq.workspace_status(ws) == goq.ERR_TIMEOUT
    assert torch.isnan(cut[2]).all() and torch.isnan(cut[3]).all()
    goq.workspace_init(ws)
    again = call()
    assert goq.workspace_status(ws) == goq.OK
    assert all(torch.equal(a, c) for a, c in zip(good, again))


@pytest.mark.parametrize("k,n,inner,m,g,b", [(256, 64, 512, 1, 64, 3), (1024, 256, 2816, 4, 128, 3), (128, 128, 256, 3, 32, 2), (4096, 1024, 11008, 4, 128, 3),
                                             (2048, 2048, 4096, 7, 128, 3), (512, 128, 1408, 2, 128, 2)])
def test_chain_shares_staged_activations(goq, k, n, inner, m, g, b):
    """Two decoder layers as a chain: q, k, v read one input, gate and up another, so their activations are staged once; linears with
    fewer records than SMs (CTAs that skip one of the sharers), ranges that need only some k-blocks, one and two activation
    buffers. Every linear against the oracle on the bits it read (fp32 sums of rounded activations, bf16 out), three launches equal."""
    from tests.gpu_util import check_bf16_output, dev, pack_weights
    shapes = [(k, k), (n, k), (n, k), (k, k), (inner, k), (inner, k), (k, inner)]
    x0 = si.bf16_activations(m, k, seed=5)
    x = dev(x0)
    items, layers, ys = [], [], []
    for layer in range(2):
        base = 7 * layer
        reads = [base - 1] * 3 + [base + (2 if n == k else 0), base + 3, base + 3, base + 5]
        for j, (no, ki) in enumerate(shapes):
            codes, meta, coef = si.random_quantized(no, ki, g, b, seed=layer * 7 + j)
            coef = (coef.astype(np.float64) * (1.5 / np.sqrt(ki)) / max(1e-9, np.std(coef.astype(np.float64)))).astype(np.float16)
            d, packed = pack_weights(no, ki, g, b, codes, meta, coef)
            y = torch.zeros((m, no), dtype=torch.bfloat16, device="cuda")
            src = reads[j]
            items.append((d, packed, x if src < 0 else ys[src], m, y, goq.BF16, False))
            layers.append((codes, meta, coef, src))
            ys.append(y)
    seq = goq.make_sequence(items)
    ws = torch.zeros(goq.sequence_workspace_bytes(len(items)), dtype=torch.uint8, device="cuda")
    runs = []
    for _ in range(3):
        for y in ys:
            y.zero_()
        goq.gemv_sequence(seq, ws)
        torch.cuda.synchronize()
        assert goq.workspace_status(ws) == goq.OK
        runs.append([y.view(torch.int16).cpu().numpy().view(np.uint16).copy() for y in ys])
    for r in runs[1:]:
        assert all(np.array_equal(a, c) for a, c in zip(runs[0], r))
    for (codes, meta, coef, src), got in zip(layers, runs[0]):
        xin = si.bf16_bits_to_f64(x0 if src < 0 else runs[0][src])
        rows = si.sample_rows(codes.shape[0], min(codes.shape[0], 64), seed=2)
        y_ref = O.linear_f64(codes, meta, coef, xin, g, b, rows=rows)
        check_bf16_output(si.bf16_bits_to_f64(got)[:, rows], y_ref, 1e-4)
