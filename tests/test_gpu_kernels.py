"""Parity of the CUDA kernels with the CPU oracle, kernel by kernel, through the C-ABI.

Integer, byte and scale-bit-pattern work must be bit-exact; dequantized fp32 outputs whose
operation order is pinned (rescale, ReLU) must be bit-exact too (tolerance 1e-6 relative is
slack); GELU outputs within 1e-6 relative with a floor of 1e-6 * max|y|; SSE within 1e-5
relative with identical rankings; bf16 layers within 1e-2 (normwise) of the fp64 reference.
"""
import numpy as np
import pytest
import torch

from oracle import qcfg_oracle as orc

pytestmark = pytest.mark.gpu

BITS = list(range(2, 9))


@pytest.fixture(scope="module")
def ctx():
    import paper_2302_01382_b200 as q
    c = q.Context(0)
    yield c
    c.close()


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def host(t):
    return t.detach().cpu().numpy()


# ----------------------------------------------------------------------------- absmax, scales

@pytest.mark.parametrize("shape", [(1, 1), (7, 13), (64, 256), (300, 768), (10, 147), (1025, 1000), (5, 40000)])
def test_absmax_matches_oracle(ctx, shape):
    import paper_2302_01382_b200 as q
    rng = np.random.default_rng(shape[0] * 1000 + shape[1])
    x = (rng.standard_normal(shape) * 10.0 ** rng.uniform(-3, 3)).astype(np.float32)
    xd = dev(x)
    np.testing.assert_array_equal(host(ctx.calibrate(xd, q.PER_TENSOR))[0], orc.absmax(x))
    np.testing.assert_array_equal(host(ctx.calibrate(xd, q.PER_ROW)), orc.absmax(x, orc.PER_ROW))
    if shape[1] > 8:  # strided, unaligned view
        v = xd[:, 3:shape[1] - 1]
        np.testing.assert_array_equal(host(ctx.calibrate(v, q.PER_TENSOR))[0], orc.absmax(x[:, 3:shape[1] - 1]))
        np.testing.assert_array_equal(host(ctx.calibrate(v, q.PER_ROW)), orc.absmax(x[:, 3:shape[1] - 1], orc.PER_ROW))
    ctx.check_sync()


def test_absmax_propagates_nonfinite_and_empty(ctx):
    import paper_2302_01382_b200 as q
    x = np.ones((4, 64), np.float32)
    x[2, 5] = np.nan
    assert not np.isfinite(host(ctx.calibrate(dev(x), q.PER_TENSOR))[0])
    x[2, 5] = -np.inf
    assert np.isinf(host(ctx.calibrate(dev(x), q.PER_ROW))[2])
    z = torch.zeros((3, 8), device="cuda")
    assert host(ctx.calibrate(z, q.PER_TENSOR))[0] == 0


@pytest.mark.parametrize("b", BITS)
def test_scales_bit_patterns(ctx, b):
    rng = np.random.default_rng(b)
    A = np.concatenate([(10.0 ** rng.uniform(-30, 30, 4000)).astype(np.float32), np.zeros(3, np.float32)])
    s, inv = ctx.scales_from_absmax(dev(A), b)
    so, io = orc.scales_from_absmax(A, b)
    np.testing.assert_array_equal(host(s).view(np.uint32), so.view(np.uint32))
    np.testing.assert_array_equal(host(inv).view(np.uint32), io.view(np.uint32))


# ----------------------------------------------------------------------------- quantize

@pytest.mark.parametrize("b", BITS)
@pytest.mark.parametrize("shape", [(3, 5), (64, 256), (257, 147), (130, 1000)])
def test_quantize_codes_bit_exact(ctx, b, shape):
    import paper_2302_01382_b200 as q
    rng = np.random.default_rng(b * 100 + shape[1])
    x = rng.standard_normal(shape).astype(np.float32)
    # exact ties and values beyond the calibrated range
    x[0, :min(5, shape[1])] = (np.arange(min(5, shape[1])) + 0.5).astype(np.float32)
    xd = dev(x)
    # per row, own maxima
    A = orc.absmax(x, orc.PER_ROW)
    so, io = orc.scales_from_absmax(A, b)
    codes = host(ctx.quantize(xd, dev(io), q.PER_ROW, b))
    np.testing.assert_array_equal(codes[:, :shape[1]], orc.quantize(x, io[:, None], b))
    assert not codes[:, shape[1]:].any()
    # per tensor, a calibrated maximum smaller than the data (live clip)
    At = np.float32(orc.absmax(x) * 0.37)
    st, it = orc.scales_from_absmax(At, b)
    codes = host(ctx.quantize(xd, dev(np.array([it], np.float32)), q.PER_TENSOR, b))
    want = orc.quantize(x, it, b)
    np.testing.assert_array_equal(codes[:, :shape[1]], want)
    assert np.abs(want).max() == orc.qmax(b)


@pytest.mark.parametrize("bits", [8, 16])
@pytest.mark.parametrize("rows", [4096, 4097])
def test_quantize_behind_other_work(ctx, rows, bits):
    """A quantize launch up to 64 MB of input is scheduled while its predecessor drains, a longer one is not: both wait
    for the kernel that writes their input."""
    import paper_2302_01382_b200 as q
    base = torch.randn((rows, 4096), device="cuda")
    inv = torch.tensor([31.0], device="cuda")
    x = torch.empty_like(base)
    for scale in (1.0, 0.25):
        torch.mul(base, scale, out=x)
        y = ctx.quantize(x, None if bits == 16 else inv, q.PER_TENSOR, bits)
        want = x.bfloat16() if bits == 16 else torch.round(x * inv).clamp(-127, 127).to(torch.int8)
        assert torch.equal(y, want)
    ctx.check_sync()


def test_quantize_bf16_bit_exact(ctx):
    import paper_2302_01382_b200 as q
    rng = np.random.default_rng(0)
    x = (rng.standard_normal((77, 203)) * 10.0 ** rng.uniform(-5, 5, (77, 1))).astype(np.float32)
    out = ctx.quantize(dev(x), None, q.PER_TENSOR, 16)
    got = host(out.float())[:, :203]
    np.testing.assert_array_equal(got.view(np.uint32), orc.bf16_round(x).view(np.uint32))


# ----------------------------------------------------------------------------- sweep

SWEEP_SHAPES = [(256, 256), (10, 256), (768, 768), (300, 3072), (97, 1024), (33, 4096), (64, 147), (128, 576),
                (40, 4608), (5, 8192), (3, 9000), (17, 64), (1, 4), (2500, 32)]


def _check_sweep(ctx, tensors, granularity):
    sse, amax = ctx.quant_error_sweep([dev(t) for t in tensors], granularity)
    ctx.check_sync()
    sse, amax = host(sse), host(amax)
    so, ao = orc.quant_error_sweep(tensors, granularity)
    np.testing.assert_array_equal(amax, ao)
    np.testing.assert_allclose(sse, so, rtol=1e-5, atol=0)
    sizes = [t.size for t in tensors]
    eg, eo = orc.e_qe_table(sse, sizes, amax), orc.e_qe_table(so, sizes, ao)
    for j in range(7):
        rg, ro = orc.ranking(eg[:, j]), orc.ranking(eo[:, j])
        if not np.array_equal(rg, ro):   # only near-ties may swap
            for a, b in zip(rg, ro):
                assert a == b or abs(eo[a, j] - eo[b, j]) <= 1e-5 * eo[a, j]


@pytest.mark.parametrize("granularity", [orc.PER_ROW, orc.PER_TENSOR])
def test_sweep_matches_oracle(ctx, granularity):
    rng = np.random.default_rng(42)
    tensors = []
    for i, s in enumerate(SWEEP_SHAPES):
        w = (rng.standard_normal(s) * 0.02).astype(np.float32)
        w[rng.random(s) < 1e-3] *= 20
        if i % 3 == 0:
            w *= rng.uniform(0.2, 5, (s[0], 1)).astype(np.float32)
        tensors.append(w)
    tensors.append(np.zeros((8, 64), np.float32))
    _check_sweep(ctx, tensors, granularity)


@pytest.mark.parametrize("granularity", [orc.PER_ROW, orc.PER_TENSOR])
@pytest.mark.parametrize("shapes,offset", [
    ([(256, 256), (10, 256)], 0),                    # fewer pieces than resident blocks
    ([(0, 64), (5, 64), (3, 0), (64, 147)], 0),      # empty tensors, rows that are not whole float4
    ([(1300, 768), (40, 3072)], 0),                  # one row kind, teams of one and of four warps
    ([(700, 1024), (77, 4096)], 0),                  # one row kind of the widest chunk
    ([(300, 768), (129, 1024), (2, 8193), (1000, 20)], 0),
    ([(130, 256), (33, 768)], 1),                    # rows that do not start on 16 bytes
])
def test_sweep_plans_match_oracle(ctx, shapes, offset, granularity):
    rng = np.random.default_rng(len(shapes) + offset)
    tensors, on_dev = [], []
    for s in shapes:
        tensors.append((rng.standard_normal(s) * rng.uniform(0.01, 3, (s[0], 1))).astype(np.float32))
        buf = torch.zeros(s[0] * s[1] + offset, device="cuda")
        buf[offset:] = dev(tensors[-1]).reshape(-1)
        on_dev.append(buf[offset:].view(s))
    for _ in range(2):                               # the second call reuses the first one's tables
        sse, amax = ctx.quant_error_sweep(on_dev, granularity)
        st, at = ctx.quant_error_sweep_static(on_dev, granularity)
        ctx.check_sync()
        full = [i for i, t in enumerate(tensors) if t.size]
        so, ao = np.zeros((len(tensors), 7)), np.zeros(len(tensors), np.float32)      # a tensor without elements: zeros
        so[full], ao[full] = orc.quant_error_sweep([tensors[i] for i in full], granularity)
        np.testing.assert_array_equal(host(amax), ao)
        np.testing.assert_allclose(host(sse), so, rtol=1e-5, atol=0)
        assert torch.equal(sse, st) and torch.equal(amax, at)


@pytest.mark.parametrize("cols,offset,terms", [(147, 0, 1), (256, 1, 1), (511, 0, 1), (513, 0, 2), (771, 0, 3)])
def test_sweep_of_ragged_rows_sums_in_64_bits(ctx, cols, offset, terms):
    """Rows that are not whole aligned float4: at most `terms` squared errors meet in fp32, so the sum is within terms * 2^-24
    of the exact sum of the rounded errors.  One row in 48 has a few errors of 0.45, all others are 7e-5: the square of
    such an error vanishes when fp32 adds it to that of a large one, so long fp32 chains lose more than that."""
    rows = 20000
    x = np.full((rows, cols), 7e-5, np.float32)
    x[::48, 1:64] = 0.45
    x[:, 0] = 1.0                                     # the row maximum: at 2 bit the grid is -1, 0, 1 and x its own error
    buf = torch.zeros(rows * cols + offset, device="cuda")
    buf[offset:] = dev(x).reshape(-1)
    e = x[:, 1:].astype(np.float64)
    want = float((e * e).sum())
    for sweep in (ctx.quant_error_sweep, ctx.quant_error_sweep_static):
        sse, _ = sweep([buf[offset:].view(rows, cols)])
        ctx.check_sync()
        assert abs(float(sse[0, 0]) - want) <= (terms * 2.0 ** -24 + 1e-12) * want


def test_sweep_is_deterministic_and_handles_subranges(ctx):
    rng = np.random.default_rng(1)
    ts = [dev((rng.standard_normal((500, 768)) * 0.02).astype(np.float32)) for _ in range(3)]
    a, _ = ctx.quant_error_sweep(ts)
    b, _ = ctx.quant_error_sweep(ts)
    assert torch.equal(a, b)
    c, _ = ctx.quant_error_sweep(ts, b_lo=4, b_hi=6)
    assert torch.equal(c, a[:, 2:5])


# ----------------------------------------------------------------------------- GEMM

def _codes(rng, rows, k, ld, lo=-127, hi=127):
    q = np.zeros((rows, ld), np.int8)
    q[:, :k] = rng.integers(lo, hi + 1, (rows, k), dtype=np.int8)
    return q


GEMM_SHAPES = [(64, 16, 32), (128, 32, 128), (64, 10, 256), (300, 200, 150), (700, 1000, 528), (129, 257, 3072),
               (1000, 768, 768), (260, 2304, 144), (3, 5, 7), (2048, 64, 64), (512, 512, 4608)]


# ragged in rows and columns and large enough that the tiles stay 256 columns wide
WIDE = [(4993, 1000), (5000, 1000), (257, 19300)]


def tile_columns(m, n):
    """Width of a single GEMM's tiles: by the output's columns, halved while every CTA still has one tile at most."""
    width = 256 if n > 128 else 128 if n > 64 else 64 if n > 32 else 32
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    while width > 32 and -(-n // (width // 2)) * -(-m // 128) <= sms:
        width //= 2
    return width


@pytest.mark.parametrize("m,n", WIDE)
def test_wide_shapes_keep_whole_tiles(m, n):
    assert tile_columns(m, n) == 256 and n % 256 and m % 256


@pytest.mark.parametrize("m,n,k", GEMM_SHAPES)
def test_gemm_i8_accumulators_and_rescale_bit_exact(ctx, m, n, k):
    import paper_2302_01382_b200 as q
    rng = np.random.default_rng(m + n + k)
    ld = (k + 15) // 16 * 16
    qx, qw = _codes(rng, m, k, ld), _codes(rng, n, k, ld)
    sw = (10.0 ** rng.uniform(-4, -2, n)).astype(np.float32)
    sx = np.float32(0.0173)
    y, acc = ctx.gemm_i8(dev(qx), dev(qw), k, float(sx), dev(sw), q.ACT_NONE, want_y=True, want_acc=True)
    ctx.check_sync()
    ref = orc.int_gemm(qx[:, :k], qw[:, :k])
    np.testing.assert_array_equal(host(acc), ref)
    np.testing.assert_array_equal(host(y).view(np.uint32), orc.dequant_output(ref, sx, sw).view(np.uint32))


@pytest.mark.parametrize("m,n,k", [(5000, 1024, 272), (257, 300, 1040), (129, 2304, 64), (4993, 1000, 272), (257, 19300, 80)])
def test_gemm_pair_and_single_cta_tiles_agree(ctx, m, n, k):
    """Outputs wider than 128 columns run on CTA pairs (256-row tiles); the single-CTA path must
    give the same bits, also when a pair works through several tiles and when the second CTA's
    rows or columns lie partly or wholly outside the matrix."""
    import paper_2302_01382_b200 as q
    rng = np.random.default_rng(m * 7 + n)
    ld = (k + 15) // 16 * 16
    qx, qw = _codes(rng, m, k, ld), _codes(rng, n, k, ld)
    sw = (10.0 ** rng.uniform(-4, -2, n)).astype(np.float32)
    res = []
    for pair in (True, False):
        ctx.set_pair_tiles(pair)
        try:
            y, acc = ctx.gemm_i8(dev(qx), dev(qw), k, 0.021, dev(sw), q.ACT_GELU_TANH, want_y=True, want_acc=True)
            ctx.check_sync()
        finally:
            ctx.set_pair_tiles(True)
        res.append((y, acc))
    np.testing.assert_array_equal(host(res[0][1]), orc.int_gemm(qx[:, :k], qw[:, :k]))
    assert torch.equal(res[0][1], res[1][1])
    assert torch.equal(res[0][0].view(torch.int32), res[1][0].view(torch.int32))


@pytest.mark.parametrize("m,n,k", [(3072, 768, 144), (2945, 641, 48), (257, 4600, 80), (129, 9000, 16), (3072, 768, 1552)])
def test_gemm_pairs_on_narrowed_tiles_match_the_reference(ctx, m, n, k):
    """Wide outputs whose tiles were narrowed to 128 columns run on pairs while each has one tile: integer sums
    are exact, and the 16-bit products give the same bits as one CTA per tile."""
    import paper_2302_01382_b200 as q
    rng = np.random.default_rng(m * 3 + n)
    ld = (k + 15) // 16 * 16
    qx, qw = _codes(rng, m, k, ld), _codes(rng, n, k, ld)
    sw = (10.0 ** rng.uniform(-4, -2, n)).astype(np.float32)
    y, acc = ctx.gemm_i8(dev(qx), dev(qw), k, 0.0173, dev(sw), q.ACT_NONE, want_y=True, want_acc=True)
    ctx.check_sync()
    ref = orc.int_gemm(qx[:, :k], qw[:, :k])
    np.testing.assert_array_equal(host(acc), ref)
    np.testing.assert_array_equal(host(y).view(np.uint32), orc.dequant_output(ref, np.float32(0.0173), sw).view(np.uint32))
    xq = ctx.quantize(dev(rng.standard_normal((m, k)).astype(np.float32)), None, q.PER_TENSOR, 16)
    wq = ctx.quantize(dev(rng.standard_normal((n, k)).astype(np.float32)), None, q.PER_TENSOR, 16)
    res = []
    for pair in (True, False):
        ctx.set_pair_tiles(pair)
        try:
            res.append(ctx.gemm_bf16(xq, wq, k))
            ctx.check_sync()
        finally:
            ctx.set_pair_tiles(True)
    assert torch.equal(res[0].view(torch.int32), res[1].view(torch.int32))


@pytest.mark.parametrize("m,n,k", [(1, 33, 16), (31, 1, 48), (257, 259, 64), (128, 255, 144), (300, 1025, 32), (33, 65, 4608)])
def test_gemm_row_pitch_without_16_byte_alignment(ctx, m, n, k):
    """fp32 and raw outputs whose rows TMA cannot write, at the edges of a 32 x 32 piece: bit-exact, and
    nothing outside the matrix is written."""
    import ctypes as C
    import paper_2302_01382_b200 as q
    rng = np.random.default_rng(m * n + k)
    ld = (k + 15) // 16 * 16
    qx, qw = _codes(rng, m, k, ld), _codes(rng, n, k, ld)
    sw = (10.0 ** rng.uniform(-4, -2, n)).astype(np.float32)
    sx = np.float32(0.0173)
    guard = 64
    y = torch.full((m * n + 2 * guard,), 7.0, device="cuda")
    acc = torch.full((m * n + 2 * guard,), 7, dtype=torch.int32, device="cuda")
    qxd, qwd, swd = dev(qx), dev(qw), dev(sw)
    for out, dst in ((y, "y"), (acc, "acc")):
        p = C.c_void_p(out.data_ptr() + 4 * guard)
        rc = ctx.lib.qcfg_gemm_i8(ctx.h, C.c_void_p(qxd.data_ptr()), ld, C.c_void_p(qwd.data_ptr()), ld, m, n, k, float(sx),
                                  C.c_void_p(swd.data_ptr()), 0, p if dst == "y" else None, p if dst == "acc" else None,
                                  C.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert rc == q.OK
    ctx.check_sync()
    want = orc.int_gemm(qx[:, :k], qw[:, :k])
    np.testing.assert_array_equal(host(acc)[guard:-guard].reshape(m, n), want)
    np.testing.assert_array_equal(host(y)[guard:-guard].reshape(m, n), orc.dequant_output(want, sx, sw))
    for out in (y, acc):
        assert (host(out)[:guard] == 7).all() and (host(out)[-guard:] == 7).all()


@pytest.mark.parametrize("m,n,k,off", [(4099, 1001, 48, 0), (6401, 259, 32, 1), (6399, 385, 80, 2), (3000, 1030, 16, 3), (38001, 255, 16, 1), (128 * 151, 257, 96, 0)])
@pytest.mark.parametrize("pair", [True, False])
def test_wide_rows_without_16_byte_pitch_are_written_line_by_line(ctx, m, n, k, off, pair):
    """256-column tiles of fp32 matrices TMA cannot write, with and without CTA pairs: row starts at every place of a
    128-byte line, last column tiles of one to 255 columns, a last row tile of one row; bit-exact against the same
    product into an aligned matrix, and nothing outside is written.  16-bit operands and GELU likewise."""
    import ctypes as C
    import paper_2302_01382_b200 as q
    rng = np.random.default_rng(m + n + k)
    ld, na = (k + 15) // 16 * 16, (n + 3) // 4 * 4
    qx, qw = _codes(rng, m, k, ld), np.zeros((na, ld), np.int8)
    qw[:n] = _codes(rng, n, k, ld)
    sw = np.ones(na, np.float32)
    sw[:n] = (10.0 ** rng.uniform(-4, -2, n)).astype(np.float32)
    st = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    ctx.set_pair_tiles(pair)
    try:
        for bf16 in (False, True):
            x, w = dev(qx), dev(qw)
            if bf16:
                x, w = x.to(torch.bfloat16) * 0.37, w.to(torch.bfloat16)
            swd = dev(sw)
            for act in (0, 2):
                res = []
                for cols, guard in ((na, 64), (n, 64 + off)):        # aligned, then the odd pitch
                    y = torch.full((m * cols + 256,), 7.0, device="cuda")
                    p = C.c_void_p(y.data_ptr() + 4 * guard)
                    xp, wp = C.c_void_p(x.data_ptr()), C.c_void_p(w.data_ptr())
                    if bf16:
                        rc = ctx.lib.qcfg_gemm_bf16(ctx.h, xp, ld, wp, ld, m, cols, k, act, p, st)
                    else:
                        rc = ctx.lib.qcfg_gemm_i8(ctx.h, xp, ld, wp, ld, m, cols, k, 0.0173, C.c_void_p(swd.data_ptr()), act, p, None, st)
                    assert rc == q.OK
                    ctx.check_sync()
                    assert (y[:guard] == 7).all() and (y[guard + m * cols:] == 7).all()
                    res.append(y[guard:guard + m * cols].reshape(m, cols)[:, :n])
                assert torch.equal(res[0].contiguous().view(torch.int32), res[1].contiguous().view(torch.int32))
    finally:
        ctx.set_pair_tiles(True)


@pytest.mark.parametrize("m,n,k,bf16,rows", [
    (10001, 175, 48, False, False), (10001, 177, 48, False, True), (10001, 207, 500, True, False), (10001, 209, 500, True, True),
    (10001, 209, 499, True, False), (12093, 2081, 16, True, False), (12100, 2081, 16, True, True)])
def test_rows_written_line_by_line_where_that_pays(ctx, m, n, k, bf16, rows):
    """Both sides of the rule that chooses the body for fp32 rows TMA cannot write: the body it names runs, with the bits of
    the same product into an aligned matrix."""
    rng = np.random.default_rng(n + k)
    ld, na = (k + 15) // 16 * 16, (n + 3) // 4 * 4
    x, w = dev(_codes(rng, m, k, ld)), torch.zeros((na, ld), dtype=torch.int8, device="cuda")
    w[:n] = dev(_codes(rng, n, k, ld))
    sw = torch.linspace(1e-4, 1e-2, na, device="cuda")
    if bf16:
        x, w = x.to(torch.bfloat16) * 0.37, w.to(torch.bfloat16)
    res = []
    for cols in (na, n):
        before = ctx.launch_forms()["rows"]
        res.append(ctx.gemm_bf16(x, w[:cols], k) if bf16 else ctx.gemm_i8(x, w[:cols], k, 0.0173, sw[:cols])[0])
        ctx.check_sync()
        assert ctx.launch_forms()["rows"] - before == (1 if rows and cols == n else 0)
    assert torch.equal(res[0][:, :n].contiguous().view(torch.int32), res[1].view(torch.int32))


@pytest.mark.parametrize("m,n,k,pairs", [(1, 32, 16, False), (129, 132, 48, False), (300, 36, 771, False), (3072, 768, 96, True), (3001, 764, 130, True),
                                         (6300, 132, 64, True), (2048, 1028, 3072, True)])
@pytest.mark.parametrize("pair", [True, False])
def test_narrow_fp32_tiles(ctx, m, n, k, pairs, pair):
    """Launches of one narrow tile per CTA with fp32 output: the bits of the general body, which a raw-accumulator output asks
    for.  Where CTA pairs apply (on 148 SMs) a lone GEMM keeps the general body."""
    import paper_2302_01382_b200 as q
    rng = np.random.default_rng(m + n + k)
    ld = (k + 15) // 16 * 16
    x, w = dev(_codes(rng, m, k, ld)), dev(_codes(rng, n, k, ld))
    sw = dev((10.0 ** rng.uniform(-4, -2, n)).astype(np.float32))
    ctx.set_pair_tiles(pair)
    try:
        for act in (q.ACT_NONE, q.ACT_RELU, q.ACT_GELU_TANH):
            before = ctx.launch_forms()["narrow_fp32"]
            y = ctx.gemm_i8(x, w, k, 0.0173, sw, act)[0]
            taken = 0 if pairs and pair else 1
            assert ctx.launch_forms()["narrow_fp32"] == before + taken
            general, acc = ctx.gemm_i8(x, w, k, 0.0173, sw, act, want_acc=True)
            assert ctx.launch_forms()["narrow_fp32"] == before + taken
            ctx.check_sync()
            assert torch.equal(y.view(torch.int32), general.view(torch.int32)) and acc.any()
    finally:
        ctx.set_pair_tiles(True)


FIRST_GEMMS = r"""
import sys
sys.path.insert(0, {root!r})
import torch
import paper_2302_01382_b200 as q
ctx = q.Context(0)
gen = torch.Generator(device="cuda")
gen.manual_seed(1)
for m, n, k in ((64, 32, 64), (1000, 1024, 256), (9000, 259, 64), (3000, 96, 64)):
    x, w = (torch.randint(-9, 10, (r, k), dtype=torch.int8, device="cuda", generator=gen) for r in (m, n))
    xb, wb, sw = x.to(torch.bfloat16), w.to(torch.bfloat16), torch.full((n,), 0.01, device="cuda")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        y, z = ctx.gemm_i8(x, w, k, 0.5, sw)[0], ctx.gemm_bf16(xb, wb, k)
    graph.replay()
    assert torch.equal(z, (x.double() @ w.double().T).float())
    assert torch.equal(y, ctx.gemm_i8(x, w, k, 0.5, sw)[0]) and y.any()
    ctx.check_sync()
"""


def test_first_gemms_of_a_process_can_be_captured():
    """Kernels are set up when a context first launches them; that may be while a stream is captured."""
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    run = subprocess.run([sys.executable, "-c", FIRST_GEMMS.format(root=root)], capture_output=True, text=True, timeout=300)
    assert run.returncode == 0, run.stderr


def test_gemm_i8_worst_case_magnitude(ctx):
    k = 4608
    qx = np.full((128, k), 127, np.int8)
    qw = np.full((32, k), -127, np.int8)
    qw[::2] = 127
    _, acc = ctx.gemm_i8(dev(qx), dev(qw), k, 1.0, None, want_y=False, want_acc=True)
    ctx.check_sync()
    np.testing.assert_array_equal(host(acc), orc.int_gemm(qx, qw))


@pytest.mark.parametrize("m,n,k", [(513, 384, 256), (5000, 1000, 256)])
@pytest.mark.parametrize("act", [1, 2])
def test_gemm_i8_activations(ctx, act, m, n, k):
    rng = np.random.default_rng(act)
    qx, qw = _codes(rng, m, k, k), _codes(rng, n, k, k)
    sw = (10.0 ** rng.uniform(-3.5, -2.5, n)).astype(np.float32)
    sx = np.float32(0.011)
    y, _ = ctx.gemm_i8(dev(qx), dev(qw), k, float(sx), dev(sw), act)
    ctx.check_sync()
    pre = orc.dequant_output(orc.int_gemm(qx, qw), sx, sw)
    ref = orc.activation(pre, act)
    if act == 1:
        np.testing.assert_array_equal(host(y), ref)
    else:
        assert np.abs(pre).max() > 3       # both tails are exercised
        np.testing.assert_allclose(host(y), ref, rtol=1e-6, atol=1e-6 * np.abs(ref).max())


@pytest.mark.parametrize("next_bits", [2, 4, 8, 16])
@pytest.mark.parametrize("m,n,k,act", [(300, 200, 150, 0), (1000, 768, 768, 1), (515, 1000, 256, 0), (260, 330, 144, 1),
                                       (5000, 1000, 150, 1)])
def test_gemm_i8_requant_codes_bit_exact(ctx, m, n, k, act, next_bits):
    rng = np.random.default_rng(m + n + k + next_bits)
    ld = (k + 15) // 16 * 16
    qx, qw = _codes(rng, m, k, ld), _codes(rng, n, k, ld)
    sw = (10.0 ** rng.uniform(-4, -2, n)).astype(np.float32)
    sx = np.float32(0.0173)
    y = orc.activation(orc.dequant_output(orc.int_gemm(qx[:, :k], qw[:, :k]), sx, sw), act)
    if next_bits == 16:
        out = ctx.gemm_i8_requant(dev(qx), dev(qw), k, float(sx), dev(sw), act, 1.0, 16)
        ctx.check_sync()
        got = host(out.float())[:, :n]
        np.testing.assert_array_equal(got.view(np.uint32), orc.bf16_round(y).view(np.uint32))
    else:
        A = np.float32(np.abs(y).max() * 0.6)            # calibrated maximum below the data: live clip
        _, inv = orc.scales_from_absmax(A, next_bits)
        out = ctx.gemm_i8_requant(dev(qx), dev(qw), k, float(sx), dev(sw), act, float(inv), next_bits)
        ctx.check_sync()
        want = orc.quantize(y, inv, next_bits)
        np.testing.assert_array_equal(host(out)[:, :n], want)
        assert np.abs(want).max() == orc.qmax(next_bits)


@pytest.mark.parametrize("m,n,k", [(64, 16, 16), (300, 200, 150), (1000, 768, 768), (129, 1000, 3072), (128, 1000, 2048), (4993, 1000, 200)])
def test_gemm_bf16_matches_fp64_reference(ctx, m, n, k):
    import paper_2302_01382_b200 as q
    rng = np.random.default_rng(m * n + k)
    x = rng.standard_normal((m, k)).astype(np.float32)
    w = (rng.standard_normal((n, k)) * 0.05).astype(np.float32)
    xq = ctx.quantize(dev(x), None, q.PER_TENSOR, 16)
    wq = ctx.quantize(dev(w), None, q.PER_TENSOR, 16)
    y = host(ctx.gemm_bf16(xq, wq, k))
    ctx.check_sync()
    ref = orc.bf16_gemm(x, w)
    assert np.linalg.norm(y - ref) / np.linalg.norm(ref) <= 1e-2
    assert np.abs(y - ref).max() <= 1e-2 * np.abs(ref).max()
    # fp32 accumulation of exact bf16 products: far tighter than the stated bound
    assert np.abs(y - ref).max() <= 1e-5 * np.abs(ref).max() * np.sqrt(k)


# ----------------------------------------------------------------------------- host-side faults

def test_argument_errors_leave_outputs_untouched(ctx):
    import paper_2302_01382_b200 as q
    x = torch.ones((4, 32), device="cuda")
    with pytest.raises(q.QcfgError) as e:
        ctx.scales_from_absmax(x[0], 9)
    assert e.value.status == q.EBITS
    with pytest.raises(q.QcfgError) as e:
        ctx.quantize(x, x[0], q.PER_TENSOR, 12)
    assert e.value.status == q.EBITS
    with pytest.raises(q.QcfgError) as e:
        ctx.quantize(x, x[0], q.PER_TENSOR, 8, ldq=40)
    assert e.value.status == q.EALIGN
    with pytest.raises(q.QcfgError) as e:
        ctx.quant_error_sweep([x], b_lo=1, b_hi=8)
    assert e.value.status == q.EBITS
    qx = torch.zeros((8, 24), dtype=torch.int8, device="cuda")
    with pytest.raises(q.QcfgError) as e:
        ctx.gemm_i8(qx, qx, 24, 1.0, x[0])
    assert e.value.status == q.EALIGN
    assert "16-byte" in ctx.last_error()
    assert ctx.sync_status() == q.OK


# ----------------------------------------------------------------------------- device-side faults

def test_bounded_wait_gives_up_and_the_context_stays_usable(ctx):
    """Device waits on a barrier that is never signalled and on counters that never advance (the
    waits of the chained GEMM launches) each run into their limit (1 ms here); only when all of
    them gave up does the kernel report QCFG_ETIMEOUT through the error word.  The context is left
    able to run a correct GEMM."""
    import paper_2302_01382_b200 as q
    assert ctx.sync_status() == q.OK
    ctx.selftest_wait_timeout(1_000_000)
    assert ctx.sync_status() == q.ETIMEOUT
    assert "wait" in ctx.last_error()
    assert ctx.sync_status() == q.OK                  # the error word was cleared by the read
    rng = np.random.default_rng(5)
    qx = rng.integers(-127, 128, (200, 64), dtype=np.int8)
    qw = rng.integers(-127, 128, (48, 64), dtype=np.int8)
    _, acc = ctx.gemm_i8(dev(qx), dev(qw), 64, 1.0, None, want_y=False, want_acc=True)
    assert ctx.sync_status() == q.OK
    np.testing.assert_array_equal(host(acc), orc.int_gemm(qx, qw))
    with pytest.raises(q.QcfgError) as e:
        ctx.selftest_wait_timeout(0)
    assert e.value.status == q.EINVAL


def test_second_context_sweeps_wide_rows():
    """The sweep's shared-memory opt-in is set per context: a context created after another one
    has already swept still runs the variants that need more than 48 KB of shared memory."""
    import paper_2302_01382_b200 as q
    rng = np.random.default_rng(6)
    x = rng.standard_normal((40, 768)).astype(np.float32)
    so, ao = orc.quant_error_sweep([x])
    for _ in range(2):
        c = q.Context(0)
        sse, amax = c.quant_error_sweep([dev(x)])
        c.check_sync()
        np.testing.assert_allclose(host(sse), so, rtol=1e-5)
        np.testing.assert_array_equal(host(amax), ao)
        c.close()


@pytest.mark.parametrize("m,n,k", [(1, 64, 32), (33, 16, 48), (300, 40, 64), (19000, 64, 64), (19072, 64, 256), (38001, 48, 96), (40000, 128, 64),
                                   (25000, 100, 160)])
def test_narrow_code_outputs_match_the_oracle(ctx, m, n, k):
    """One int8 code matrix of fewer than 256 columns: one to several tiles per CTA, odd and even tile counts (the 64-column
    tiles are shared out between two halves of the epilogue warps), ragged rows and columns; every code is checked."""
    import paper_2302_01382_b200 as q
    rng = np.random.default_rng(m + n + k)
    qx = rng.integers(-127, 128, (m, k), dtype=np.int8)
    qw = rng.integers(-127, 128, (n, k), dtype=np.int8)
    sw = (10.0 ** rng.uniform(-4, -2, n)).astype(np.float32)
    y = orc.activation(orc.dequant_output(orc.int_gemm(qx, qw), np.float32(0.0173), sw), orc.ACT_RELU)
    _, inv = orc.scales_from_absmax(np.float32(np.abs(y).max() * 0.6), 6)
    out = ctx.gemm_i8_requant(dev(qx), dev(qw), k, 0.0173, dev(sw), q.ACT_RELU, float(inv), 6)
    ctx.check_sync()
    np.testing.assert_array_equal(host(out)[:, :n], orc.quantize(y, inv, 6))
    assert not host(out)[:, n:].any()


@pytest.mark.parametrize("m,n,act", [(4099, 1000, 0), (9000, 520, 2), (2600, 2056, 1)])
def test_wide_bf16_outputs_match_the_oracle(ctx, m, n, act):
    """16-bit operands for the next layer out of 256-column tiles, ragged rows and columns, several tiles per CTA."""
    rng = np.random.default_rng(m + n)
    k = 96
    qx, qw = _codes(rng, m, k, k), _codes(rng, n, k, k)
    sw = (10.0 ** rng.uniform(-4, -2, n)).astype(np.float32)
    y = orc.activation(orc.dequant_output(orc.int_gemm(qx, qw), np.float32(0.0173), sw), act)
    out = ctx.gemm_i8_requant(dev(qx), dev(qw), k, 0.0173, dev(sw), act, 1.0, 16)
    ctx.check_sync()
    got, want = host(out.float())[:, :n], orc.bf16_round(y)
    if act == 2:      # GELU outputs are within 1e-6 relative plus 1e-6 * max|y| of the oracle's: rounded, between the bounds' roundings
        d = (1e-6 * np.abs(y) + 1e-6 * np.abs(y).max()).astype(np.float32)
        assert np.all(got >= orc.bf16_round(y - d)) and np.all(got <= orc.bf16_round(y + d))
    else:
        np.testing.assert_array_equal(got.view(np.uint32), want.view(np.uint32))
    assert not host(out.float())[:, n:].any()


def test_calibration_ranges_do_not_depend_on_the_route(ctx):
    """Maxima taken in the epilogue that writes the 16-bit operand equal those of separate passes, at sizes whose GEMMs
    run in 256-column tiles and in chains."""
    import paper_2302_01382_b200 as q
    import qcfg_workloads as wl
    w = wl.bert_stack(6, 9001, 392, 1544, 2, bit_choices=None)
    weights, x = [dev(a) for a in w.weights], dev(w.x)
    tables = []
    for fuse, chains in ((True, True), (True, False), (False, False)):
        ctx.set_fusion(fuse)
        ctx.set_gemm_chains(chains)
        try:
            model = q.Model(ctx, w.layers, weights)
            model.calibrate_model(x, w.m)
            tables.append(model.act_absmax())
            model.close()
        finally:
            ctx.set_fusion(True)
            ctx.set_gemm_chains(True)
    assert tables[0] == tables[1] == tables[2]
