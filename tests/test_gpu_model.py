"""Parity of whole configuration evaluations with the CPU oracle, through the C-ABI.

Primary gate: layer-wise teacher forcing.  For every layer the test downloads the fp32
input the GPU actually fed to it, lets the oracle recompute scale, codes, int32 accumulators
and output from that input, and requires codes, scale bit patterns and accumulators to be
bit-exact, outputs to be bit-exact (no activation / ReLU), within 1e-6 relative with a floor
of 1e-6 * max|y| (GELU), or within 1e-2 normwise (16-bit layers).  End-to-end chained outputs
are compared with float tolerances; the ReLU-only integer model must be bit-exact end to end.
"""
import numpy as np
import pytest
import torch

import qcfg_workloads as wl
from oracle import qcfg_oracle as orc

pytestmark = pytest.mark.gpu


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


def build(ctx, w):
    import paper_2302_01382_b200 as q
    weights = [dev(a) for a in w.weights]
    model = q.Model(ctx, w.layers, weights)
    x = dev(w.x.reshape(w.x.shape[0], -1) if w.x.ndim == 2 else w.x)
    model.calibrate_model(x, w.m)
    return model, x


def run_eval(ctx, model, w, x, bits):
    ys = [torch.full((wl.layer_rows(w.layers, l, w.m), lay.n_out), float("nan"), device="cuda")
          for l, lay in enumerate(w.layers)]
    model.eval_config(bits, x, w.m, ys)
    ctx.check_sync()
    return ys


def check_calibration(model, w):
    act_o, w_o = orc.calibrate_model(w.layers, w.weights, w.x)
    act_g = np.array(model.act_absmax(), np.float32)
    # the 16-bit forward accumulates in fp32 on the GPU and fp64 in the oracle: maxima agree to
    # bf16-product accumulation accuracy, not bit for bit (except for external inputs)
    for l, lay in enumerate(w.layers):
        if lay.src < 0 and lay.pool_before == 0:
            assert act_g[l] == act_o[l]
        else:
            assert act_g[l] == pytest.approx(float(act_o[l]), rel=2e-3)
        np.testing.assert_array_equal(np.array(model.weight_absmax(l), np.float32), w_o[l])
    return act_g, w_o


def teacher_forced_check(ctx, model, w, x, bits, ys, act_g, w_amax, sample_rows=None):
    outs = [host(y) for y in ys]
    for o in outs:
        assert np.all(np.isfinite(o)), "an output element was never written"
    for l, lay in enumerate(w.layers):
        b = int(bits[l])
        xin = orc.layer_input(w.layers, l, w.x, outs)          # built from the GPU's own outputs
        res = outs[lay.residual_from] if lay.residual_from >= 0 else None
        rows = None
        if sample_rows is not None and outs[l].shape[0] > sample_rows:
            rows = np.sort(np.random.default_rng(l).choice(outs[l].shape[0], sample_rows, replace=False))
        y_ref, taps = orc.eval_layer_teacher_forced(lay, w.weights[l], xin, b, act_g[l], w_amax[l], residual=res, rows=rows)
        y_gpu = outs[l] if rows is None else outs[l][rows]
        if b == 16:
            assert np.linalg.norm(y_gpu - y_ref) <= 1e-2 * max(np.linalg.norm(y_ref), 1e-30), l
            assert np.abs(y_gpu - y_ref).max() <= 1e-2 * max(np.abs(y_ref).max(), 1e-30), l
            continue
        m_rows, k = outs[l].shape[0], lay.k_in
        qx = torch.empty((m_rows, k), dtype=torch.int8, device="cuda")
        qw = torch.empty((lay.n_out, k), dtype=torch.int8, device="cuda")
        acc = torch.empty((m_rows, lay.n_out), dtype=torch.int32, device="cuda")
        model.debug_dump(l, qx, qw, acc)
        ctx.check_sync()
        qx, acc = host(qx), host(acc)
        if rows is not None:
            qx, acc = qx[rows], acc[rows]
        np.testing.assert_array_equal(qx, taps["qx"], err_msg=f"layer {l} input codes")
        np.testing.assert_array_equal(host(qw), taps["qw"], err_msg=f"layer {l} weight codes")
        np.testing.assert_array_equal(acc, taps["acc"], err_msg=f"layer {l} accumulators")
        if lay.act == orc.ACT_GELU_TANH:
            np.testing.assert_allclose(y_gpu, y_ref, rtol=1e-6, atol=1e-6 * np.abs(y_ref).max(), err_msg=f"layer {l}")
        else:
            np.testing.assert_array_equal(y_gpu.view(np.uint32), y_ref.view(np.uint32), err_msg=f"layer {l}")


def test_tiny_mlp_bit_exact_end_to_end(ctx):
    w = wl.tiny_mlp()
    model, x = build(ctx, w)
    act_g, w_amax = check_calibration(model, w)
    ys = run_eval(ctx, model, w, x, w.bits)
    teacher_forced_check(ctx, model, w, x, w.bits, ys, act_g, w_amax)
    # chained oracle with the GPU's calibration table: integers and ReLU only -> bit-exact
    outs = orc.eval_config(w.layers, w.weights, w.bits, w.x, list(act_g), w_amax)
    for l in range(3):
        np.testing.assert_array_equal(host(ys[l]), outs[l])
    model.close()


@pytest.mark.parametrize("fuse", [True, False])
@pytest.mark.parametrize("seed,m,hidden,ffn,blocks", [(11, 300, 192, 768, 2), (12, 1100, 256, 1024, 1)])
def test_bert_stack_teacher_forced(ctx, fuse, seed, m, hidden, ffn, blocks):
    ctx.set_fusion(fuse)
    try:
        w = wl.bert_stack(seed, m, hidden, ffn, blocks)
        model, x = build(ctx, w)
        act_g, w_amax = check_calibration(model, w)
        for bits in (w.bits, [8] * len(w.layers), [4, 8, 16, 3, 16, 2] * blocks):
            ys = run_eval(ctx, model, w, x, bits)
            teacher_forced_check(ctx, model, w, x, bits, ys, act_g, w_amax)
            # end to end against the chained oracle: float tolerance only (GELU, bf16 layers)
            outs = orc.eval_config(w.layers, w.weights, bits, w.x, list(act_g), w_amax)
            last = host(ys[-1])
            assert np.linalg.norm(last - outs[-1]) <= 2e-2 * np.linalg.norm(outs[-1])
        model.close()
    finally:
        ctx.set_fusion(True)


@pytest.mark.parametrize("fuse", [True, False])
def test_column_slice_consumers_teacher_forced(ctx, fuse):
    """One wide projection layer (3h output channels) whose column thirds are read by three
    consumers through src_col0 = 0, h, 2h: calibration maxima, input codes, accumulators and
    outputs of every slice reader against the oracle, and the wide layer's thirds against three
    separate projections with the same weight rows."""
    ctx.set_fusion(fuse)
    try:
        h, ffn, m = 192, 768, 333
        w = wl.bert_stack_wide_qkv(33, m, h, ffn, 2)
        model, x = build(ctx, w)
        act_g, w_amax = check_calibration(model, w)
        for bits in (w.bits, [8] * len(w.layers), [4, 8, 16, 3, 16, 2] * 2, [16, 8, 4, 8, 8, 8] * 2):
            ys = run_eval(ctx, model, w, x, bits)
            teacher_forced_check(ctx, model, w, x, bits, ys, act_g, w_amax)
        ys8 = run_eval(ctx, model, w, x, [8] * len(w.layers))
        model.close()
        # all-8: the wide layer's thirds equal three separate projections
        sep = wl.Workload("sep", 33, wl.bert_layers(h, ffn, 2), m, w.x, [], bits=np.full(12, 8, np.uint8))
        for blk in range(2):
            wide = w.weights[6 * blk]
            sep.weights += [wide[:h], wide[h:2 * h], wide[2 * h:]] + w.weights[6 * blk + 3:6 * blk + 6]
        model_s, xs = build(ctx, sep)
        ys_s = run_eval(ctx, model_s, sep, xs, sep.bits)
        for blk in range(2):
            for j in range(3):
                assert torch.equal(ys8[6 * blk][:, j * h:(j + 1) * h], ys_s[6 * blk + j])
            for j in (3, 4, 5):
                assert torch.equal(ys8[6 * blk + j], ys_s[6 * blk + j])
        model_s.close()
    finally:
        ctx.set_fusion(True)


def test_fused_and_unfused_agree_bitwise_and_taps_are_optional(ctx):
    w = wl.bert_stack(21, 515, 128, 512, 2, bit_choices=(4, 8))
    model, x = build(ctx, w)
    ys_f = run_eval(ctx, model, w, x, w.bits)
    ctx.set_fusion(False)
    ys_u = run_eval(ctx, model, w, x, w.bits)
    ctx.set_fusion(True)
    for a, b in zip(ys_f, ys_u):
        assert torch.equal(a, b)
    # only the last layer requested: same values
    ys = [None] * (len(w.layers) - 1) + [torch.empty_like(ys_f[-1])]
    model.eval_config(w.bits, x, w.m, ys)
    ctx.check_sync()
    assert torch.equal(ys[-1], ys_f[-1])
    model.eval_config(w.bits, x, w.m, None)
    ctx.check_sync()
    model.close()


@pytest.mark.parametrize("bits_kind", ["uniform8", "mixed_int", "with16"])
def test_grouped_and_single_launches_agree_bitwise(ctx, bits_kind):
    """The three projections of a block read one input: when their GEMMs have the same shape and
    operand type they run as one grouped launch (also with different bit widths, i.e. different
    input codes and scales per group); a 16-bit layer among them splits the group."""
    w = wl.bert_stack(23, 700, 256, 1024, 2, bit_choices=(4, 8))
    n = len(w.layers)
    bits = {"uniform8": [8] * n, "mixed_int": [4, 8, 6, 8, 3, 8] * 2, "with16": [8, 16, 8, 4, 16, 8] * 2}[bits_kind]
    model, x = build(ctx, w)
    res = []
    for grouping in (True, False):
        ctx.set_grouping(grouping)
        try:
            ys = run_eval(ctx, model, w, x, bits)
        finally:
            ctx.set_grouping(True)
        res.append(ys)
    for a, b in zip(*res):
        assert torch.equal(a.view(torch.int32), b.view(torch.int32))
    act_g = np.array(model.act_absmax(), np.float32)
    w_amax = [np.array(model.weight_absmax(l), np.float32) for l in range(n)]
    teacher_forced_check(ctx, model, w, x, bits, res[0], act_g, w_amax)
    model.close()


def test_model_argument_errors(ctx):
    import paper_2302_01382_b200 as q
    w = wl.tiny_mlp()
    weights = [dev(a) for a in w.weights]
    model = q.Model(ctx, w.layers, weights)
    x = dev(w.x)
    with pytest.raises(q.QcfgError) as e:
        model.eval_config(w.bits, x, w.m)
    assert e.value.status == q.ESTATE
    model.calibrate_model(x, w.m)
    with pytest.raises(q.QcfgError) as e:
        model.eval_config([8, 9, 8], x, w.m)
    assert e.value.status == q.EBITS
    bad = [wl.Layer("a", 8, 16), wl.Layer("b", 8, 16, src=0)]      # reads 16 columns of an 8-wide output
    with pytest.raises(q.QcfgError) as e:
        q.Model(ctx, bad, [torch.zeros((8, 16), device="cuda")] * 2)
    assert e.value.status == q.ESHAPE
    xn = x.clone()
    xn[3, 3] = float("nan")
    with pytest.raises(q.QcfgError) as e:
        model.calibrate_model(xn, w.m)
    assert e.value.status == q.ENONFINITE
    model.close()


@pytest.mark.parametrize("fuse", [True, False])
def test_resnet_small_teacher_forced(ctx, fuse):
    """Convolutional table at reduced size: im2col operands (3-channel 7x7/2 stem, 3x3 with stride 1
    and 2, 1x1 with stride 1 and 2), max-pool, shortcuts, global average pool, 16-bit stem and fc."""
    ctx.set_fusion(fuse)
    try:
        w = wl.resnet50(seed=3, batch=3, in_hw=64, width=16, n_classes=10, blocks=(2, 1, 2, 1))
        model, x = build(ctx, w)
        act_g, w_amax = check_calibration(model, w)
        for bits in (w.bits, [8] * len(w.layers)):
            ys = run_eval(ctx, model, w, x, bits)
            teacher_forced_check(ctx, model, w, x, bits, ys, act_g, w_amax)
        outs = orc.eval_config(w.layers, w.weights, w.bits, w.x, list(act_g), w_amax)
        last = host(ys[-1])
        ref_all8 = orc.eval_config(w.layers, w.weights, [8] * len(w.layers), w.x, list(act_g), w_amax)
        assert np.linalg.norm(last - ref_all8[-1]) <= 2e-2 * np.linalg.norm(ref_all8[-1])
        model.close()
    finally:
        ctx.set_fusion(True)


@pytest.mark.parametrize("fuse", [True, False])
def test_implicit_and_materialised_convolutions_agree_bitwise(ctx, fuse):
    """The GEMM that gathers its patches from the input's NHWC codes gives, layer by layer, the same
    bits as the GEMM on a materialised patch matrix: 3x3 with stride 1 and 2, strided 1x1, channel
    counts of one to several 16-byte chunks, int8 and 16-bit layers, ragged last row tiles."""
    for width, batch, hw in ((16, 3, 64), (48, 2, 40)):
        w = wl.resnet50(seed=5, batch=batch, in_hw=hw, width=width, n_classes=10, blocks=(2, 1, 1, 1))
        model, x = build(ctx, w)
        model.calibrate_model(x, w.m)
        n = len(w.layers)
        with16 = np.array(w.bits).copy()
        with16[3::4] = 16
        for bits in (w.bits, [8] * n, with16):
            outs = {}
            for implicit in (True, False):
                ctx.set_implicit_conv(implicit)
                ctx.set_fusion(fuse)
                ys = run_eval(ctx, model, w, x, bits)
                outs[implicit] = [host(y) for y in ys]
            for l in range(n):
                np.testing.assert_array_equal(outs[True][l].view(np.uint32), outs[False][l].view(np.uint32),
                                              err_msg=f"width {width} layer {l} ({w.layers[l].name})")
        ctx.set_implicit_conv(True)
        ctx.set_fusion(True)
        model.close()


@pytest.mark.parametrize("m", [19200, 19000])
def test_chained_and_separate_launches_agree_bitwise(ctx, m):
    """A forward pass whose GEMMs go to the device as chains (one cooperative launch for up to sixteen
    consecutive GEMMs, tiles started by per-row-tile counters; a GEMM joins a chain only if it has at
    least one tile per CTA pair, hence the row counts) gives the same bits as one launch
    per GEMM: all-int8, a mix with 4-bit and 16-bit layers (both operand types chain), every
    output requested (general epilogue) and only the last one (fast epilogue bodies), whole and
    ragged last row tiles.  The launch counter shows that the chains were in fact used."""
    w = wl.bert_stack(11, m, 256, 1024, 3, bit_choices=None)
    model, x = build(ctx, w)
    n = len(w.layers)
    mixed = [16 if i % 5 == 4 else (4 if i % 3 == 0 else 8) for i in range(n)]
    last = torch.empty((m, w.layers[-1].n_out), device="cuda")
    try:
        for bits in ([8] * n, mixed, [16] * n):
            outs, lasts, launches = {}, {}, {}
            for chained in (True, False):
                ctx.set_gemm_chains(chained)
                ys = run_eval(ctx, model, w, x, bits)
                outs[chained] = [host(y) for y in ys]
                last.fill_(float("nan"))
                n0 = ctx.launch_count()
                model.eval_config(bits, x, m, [None] * (n - 1) + [last])
                ctx.check_sync()
                launches[chained] = ctx.launch_count() - n0
                lasts[chained] = host(last).copy()
            for l in range(n):
                np.testing.assert_array_equal(outs[True][l].view(np.uint32), outs[False][l].view(np.uint32),
                                              err_msg=f"layer {l} ({w.layers[l].name}) bits {bits[l]}")
            np.testing.assert_array_equal(lasts[True].view(np.uint32), lasts[False].view(np.uint32))
            assert np.all(np.isfinite(lasts[True]))
            assert launches[True] < launches[False], launches
    finally:
        ctx.set_gemm_chains(True)
        model.close()


def test_calibration_maxima_do_not_depend_on_fusion_or_chaining(ctx):
    """The calibration forward may take an activation's range in the epilogue of the GEMM that
    produces it (fusion on: the 16-bit operand codes come from there too, and the GEMMs chain) or in
    the kernel that builds the 16-bit operand (fusion off).  Both read the same fp32 values and fold
    bit patterns with an integer maximum, so the tables agree bit for bit."""
    w = wl.bert_stack(5, 19200, 256, 1024, 2, bit_choices=None)
    model, x = build(ctx, w)
    try:
        tables = {}
        for fuse in (True, False):
            for chained in (True, False):
                ctx.set_fusion(fuse)
                ctx.set_gemm_chains(chained)
                model.calibrate_model(x, w.m)
                tables[(fuse, chained)] = np.array(model.act_absmax(), np.float32)
        ref = tables[(False, False)]
        assert np.all(ref > 0)
        for key, t in tables.items():
            np.testing.assert_array_equal(t.view(np.uint32), ref.view(np.uint32), err_msg=str(key))
    finally:
        ctx.set_fusion(True)
        ctx.set_gemm_chains(True)
        model.close()


@pytest.mark.parametrize("m,n", [(1, 32), (127, 36), (130, 100), (257, 128), (300, 132), (1200, 388), (40000, 256)])
def test_shortcut_layers_at_tile_edges(ctx, m, n):
    """Layers with an fp32 shortcut whose result goes to the caller and, as codes of two grids, to two readers:
    rows and columns at the edges of tiles and of 32 x 32 blocks, one to many tiles per CTA."""
    L = wl.Layer
    layers = [L("a", n, 48, src=-1), L("b", n, n, src=0, act=orc.ACT_RELU, residual_from=0), L("c", 16, n, src=1), L("d", 24, n, src=1),
              L("e", n, 24, src=3, residual_from=1)]
    rng = np.random.default_rng(m + n)
    x = rng.standard_normal((m, 48)).astype(np.float32)
    ws = [(rng.standard_normal((l.n_out, l.k_in)) / np.sqrt(l.k_in)).astype(np.float32) for l in layers]
    w = wl.Workload("shortcut", 1, layers, m, x, ws)
    model, xd = build(ctx, w)
    act_g, w_amax = check_calibration(model, w)
    for bits in ([8, 6, 8, 4, 8], [8, 8, 4, 4, 16]):
        ys = run_eval(ctx, model, w, xd, bits)
        teacher_forced_check(ctx, model, w, xd, bits, ys, act_g, w_amax, sample_rows=300)
        only = [None] * 4 + [torch.full_like(ys[4], float("nan"))]        # shortcuts and readers inside the model
        model.eval_config(bits, xd, m, only)
        ctx.check_sync()
        assert torch.equal(only[4], ys[4])
    model.close()


@pytest.mark.parametrize("m,n", [(9001, 516), (2500, 1156), (20000, 132)])
def test_shortcut_tiles_column_tile_fastest(ctx, m, n):
    """Shortcut layers of several column tiles and more tiles than SMs, so that a CTA's steps wrap in both coordinates: output
    and codes of the body of their own are those of the general one (which a raw-accumulator tap asks for) on every row."""
    L = wl.Layer
    layers = [L("a", n, 32, src=-1), L("b", n, 64, src=-1, src_col0=32, act=orc.ACT_RELU, residual_from=0), L("c", 16, n, src=1)]
    rng = np.random.default_rng(m + n)
    x = rng.standard_normal((m, 96)).astype(np.float32)
    ws = [(rng.standard_normal((l.n_out, l.k_in)) / np.sqrt(l.k_in)).astype(np.float32) for l in layers]
    w = wl.Workload("shortcut", 1, layers, m, x, ws)
    model, xd = build(ctx, w)
    act_g, w_amax = check_calibration(model, w)
    before = ctx.launch_forms()["shortcut"]
    ys = run_eval(ctx, model, w, xd, [8, 6, 8])
    assert ctx.launch_forms()["shortcut"] == before + 1
    teacher_forced_check(ctx, model, w, xd, [8, 6, 8], ys, act_g, w_amax)
    model.close()


@pytest.mark.parametrize("pair", [True, False])
@pytest.mark.parametrize("m,hidden", [(3072, 256), (2900, 200), (300, 64)])
def test_narrow_fp32_groups_beside_a_general_body(ctx, m, hidden, pair):
    """Projections in one grouped launch of narrow tiles: those that only return fp32 run in the straight-line body, the one
    that also feeds a reader in the general one, with and without CTA pairs."""
    L = wl.Layer
    layers = [L("q", hidden, 96, src=-1), L("k", hidden, 96, src=-1), L("v", hidden, 96, src=-1), L("o", hidden, hidden, src=2)]
    rng = np.random.default_rng(m)
    x = rng.standard_normal((m, 96)).astype(np.float32)
    ws = [(rng.standard_normal((l.n_out, l.k_in)) / np.sqrt(l.k_in)).astype(np.float32) for l in layers]
    w = wl.Workload("groups", 1, layers, m, x, ws)
    model, xd = build(ctx, w)
    act_g, w_amax = check_calibration(model, w)
    ctx.set_pair_tiles(pair)
    try:
        for bits in ([8, 8, 8, 8], [4, 8, 6, 3]):
            before = ctx.launch_forms()["narrow_fp32"]
            ys = run_eval(ctx, model, w, xd, bits)
            assert ctx.launch_forms()["narrow_fp32"] == before + 3
            teacher_forced_check(ctx, model, w, xd, bits, ys, act_g, w_amax)
    finally:
        ctx.set_pair_tiles(True)
    model.close()


@pytest.mark.parametrize("m,n,k,act", [(300, 200, 768, 2), (300, 200, 784, 2), (257, 132, 2064, 2), (9000, 260, 1280, 2), (9000, 260, 1296, 1),
                                       (33000, 36, 1024, 2), (130, 48, 64, 2)])
def test_shortcut_layers_of_long_reductions(ctx, m, n, k, act):
    """Short reductions have a shortcut body of their own, long ones the general one (the line depends on the reduction and
    on the number of tiles): both sides of it, with GELU behind the shortcut."""
    L = wl.Layer
    layers = [L("a", n, 32, src=-1), L("b", n, k, src=-1, act=act, residual_from=0), L("c", 16, n, src=1), L("d", 24, n, src=1)]
    rng = np.random.default_rng(m + n + k)
    x = rng.standard_normal((m, k)).astype(np.float32)
    ws = [(rng.standard_normal((l.n_out, l.k_in)) / np.sqrt(l.k_in)).astype(np.float32) for l in layers]
    w = wl.Workload("shortcut", 1, layers, m, x, ws)
    model, xd = build(ctx, w)
    act_g, w_amax = check_calibration(model, w)
    bits = [8, 8, 6, 4]
    ys = run_eval(ctx, model, w, xd, bits)
    teacher_forced_check(ctx, model, w, xd, bits, ys, act_g, w_amax, sample_rows=200)
    model.close()


def test_shortcut_behind_a_long_reduction_stays_in_its_chain(ctx):
    """A wide layer with a shortcut and a reduction of 1536 runs in the same chained launch as its producers; one that
    does not, takes a launch of its own."""
    L = wl.Layer
    m, n = 4992, 1536
    weights = [torch.randn((n, n), device="cuda") / n ** 0.5 for _ in range(3)]
    x = torch.randn((m, n), device="cuda")
    y = torch.empty((m, n), device="cuda")
    launches = []
    for residual in (-1, 0):
        import paper_2302_01382_b200 as q
        layers = [L("a", n, n, src=-1), L("b", n, n, src=0), L("c", n, n, src=1, residual_from=residual)]
        model = q.Model(ctx, layers, weights)
        model.calibrate_model(x, m)
        model.eval_config([8] * 3, x, m, [None, None, y])
        before = ctx.launch_count()
        model.eval_config([8] * 3, x, m, [None, None, y])
        launches.append(ctx.launch_count() - before)
        ctx.check_sync()
        model.close()
    assert launches[0] == launches[1]


@pytest.mark.parametrize("c,n,hw,k,stride,pad,batch", [(64, 64, 9, 3, 1, 1, 3), (64, 256, 13, 3, 1, 1, 5), (128, 128, 14, 3, 2, 1, 4),
                                                       (192, 48, 7, 3, 2, 1, 7), (128, 512, 8, 1, 2, 0, 33), (64, 32, 11, 5, 1, 2, 2),
                                                       (64, 64, 130, 3, 1, 0, 1), (256, 256, 4, 3, 1, 1, 40),
                                                       (64, 264, 27, 3, 1, 1, 9), (128, 264, 28, 3, 1, 1, 9)])
def test_convolution_operand_through_tma_matches_the_patch_matrix(ctx, c, n, hw, k, stride, pad, batch):
    """Channels in whole 64- and 128-byte chunks: TMA brings the patches.  Filters of one, nine and 25 taps (odd chunk
    counts leave half a k-block), strides, tiles that cross rows and images, a ragged last tile; 264 columns on more than 6400
    rows: CTA pairs, whose tiles stay 256 columns wide and whose last one is ragged."""
    L = wl.Layer
    oh = (hw + 2 * pad - k) // stride + 1
    layers = [L("in", c, 16, src=-1, kh=1, kw=1, stride=1, in_h=hw, in_w=hw, in_c=16, src_h=hw, src_w=hw),
              L("conv", n, k * k * c, src=0, act=orc.ACT_RELU, kh=k, kw=k, stride=stride, pad=pad, in_h=hw, in_w=hw, in_c=c, src_h=hw, src_w=hw),
              L("out", 16, n, src=1, kh=1, kw=1, stride=1, in_h=oh, in_w=oh, in_c=n, src_h=oh, src_w=oh)]
    rng = np.random.default_rng(c + n + hw)
    x = rng.standard_normal((batch, hw, hw, 16)).astype(np.float32)
    ws = [(rng.standard_normal((l.n_out, l.k_in)) / np.sqrt(l.k_in)).astype(np.float32) for l in layers]
    w = wl.Workload("conv", 1, layers, batch, x, ws)
    model, xd = build(ctx, w)
    act_g, w_amax = check_calibration(model, w)
    for bits in ([8, 8, 8], [8, 5, 16], [8, 16, 4]):
        outs = []
        for implicit in (True, False):
            ctx.set_implicit_conv(implicit)
            outs.append(run_eval(ctx, model, w, xd, bits))
            if implicit:
                teacher_forced_check(ctx, model, w, xd, bits, outs[0], act_g, w_amax)
        ctx.set_implicit_conv(True)
        for a, b in zip(*outs):
            assert torch.equal(a, b)
    model.close()


@pytest.mark.parametrize("c,k,hw", [(32, 3, 9), (32, 5, 11), (64, 3, 10), (48, 3, 9)])
def test_non_finite_convolution_inputs_reach_only_their_windows(ctx, c, k, hw):
    """16-bit convolutions of an input with infinities and NaN, gathered and from a patch matrix: the same outputs, where
    an odd number of 64-byte chunks leaves half a k-block empty (32 channels) and where it does not."""
    L = wl.Layer
    pad, batch = k // 2, 3
    geo = dict(kh=k, kw=k, stride=1, pad=pad, in_h=hw, in_w=hw, src_h=hw, src_w=hw)
    layers = [L("in", c, 16, src=-1, kh=1, kw=1, stride=1, in_h=hw, in_w=hw, in_c=16, src_h=hw, src_w=hw),
              L("conv", 48, k * k * c, src=0, in_c=c, **geo)]
    rng = np.random.default_rng(c + k)
    x = rng.standard_normal((batch, hw, hw, 16)).astype(np.float32)
    ws = [(rng.standard_normal((l.n_out, l.k_in)) / np.sqrt(l.k_in)).astype(np.float32) for l in layers]
    ws[0][:] = 0.0
    ws[0][:, 0] = 1.0                                     # every channel is the input's first one
    ws[1] = np.abs(ws[1])                                 # an infinity in a window stays one
    w = wl.Workload("conv", 1, layers, batch, x, ws)
    model, xd = build(ctx, w)
    check_calibration(model, w)
    xd[0, 0, 0, 0], xd[1, hw // 2, 3, 0], xd[2, hw - 1, hw - 1, 0] = float("inf"), float("nan"), float("-inf")
    outs = []
    for implicit in (True, False):
        ctx.set_implicit_conv(implicit)
        outs.append(host(run_eval(ctx, model, w, xd, [16, 16])[1]).reshape(batch, hw, hw, 48))
    ctx.set_implicit_conv(True)
    np.testing.assert_array_equal(outs[0], outs[1])
    assert np.isinf(outs[0]).any()
    oy, ox = np.mgrid[:hw, :hw]
    for b, y, z in ((0, 0, 0), (1, hw // 2, 3), (2, hw - 1, hw - 1)):
        touched = (abs(oy - y) <= pad) & (abs(ox - z) <= pad)
        assert np.isfinite(outs[0][b][~touched]).all() and not np.isfinite(outs[0][b][touched]).any()
    model.close()


@pytest.mark.parametrize("c,n,h,wd,k,pad,batch,act", [(3, 64, 32, 32, 7, 3, 3, 1), (3, 32, 33, 47, 7, 3, 2, 1), (1, 16, 20, 9, 5, 2, 40, 0),
                                                      (4, 48, 17, 255, 3, 1, 2, 1), (2, 64, 7, 8, 7, 0, 5, 0), (3, 64, 65, 224, 7, 3, 4, 1),
                                                      (3, 16, 16, 64, 8, 3, 2, 1), (3, 64, 16, 260, 7, 3, 1, 1), (5, 64, 16, 16, 3, 1, 2, 1)])
def test_stem_and_its_pool_match_the_oracle(ctx, c, n, h, wd, k, pad, batch, act):
    """Stride-2 convolutions of few channels at 16 bit with max-pooled readers: odd and even sizes and paddings, one to
    four channels, rows up to the widest, many images, and geometries the stem kernel leaves to the general path.  The
    pooled values must be the maxima of the very outputs the layer returns (its readers' integer outputs are checked
    bit for bit), and the readers' results must not depend on whether the full output is returned."""
    L = wl.Layer
    oh, ow = (h + 2 * pad - k) // 2 + 1, (wd + 2 * pad - k) // 2 + 1
    ph, pw = (oh + 2 - 3) // 2 + 1, (ow + 2 - 3) // 2 + 1
    layers = [L("stem", n, k * k * c, src=-1, act=act, kh=k, kw=k, stride=2, pad=pad, in_h=h, in_w=wd, in_c=c, src_h=h, src_w=wd),
              L("a", 24, n, src=0, kh=1, kw=1, stride=1, in_h=ph, in_w=pw, in_c=n, pool_before=wl.POOL_MAX3S2, src_h=oh, src_w=ow),
              L("b", 16, n, src=0, kh=1, kw=1, stride=1, in_h=ph, in_w=pw, in_c=n, pool_before=wl.POOL_MAX3S2, src_h=oh, src_w=ow)]
    rng = np.random.default_rng(h * wd + n)
    x = rng.standard_normal((batch, h, wd, c)).astype(np.float32)
    ws = [(rng.standard_normal((l.n_out, l.k_in)) / np.sqrt(l.k_in)).astype(np.float32) for l in layers]
    w = wl.Workload("stem", 1, layers, batch, x, ws)
    model, xd = build(ctx, w)
    act_g, w_amax = check_calibration(model, w)
    bits = [16, 8, 5]
    ys = run_eval(ctx, model, w, xd, bits)
    teacher_forced_check(ctx, model, w, xd, bits, ys, act_g, w_amax)
    # fp32 sums of exact bf16 products: each within K rounding steps of the magnitude sum
    ref = orc.bf16_gemm(orc.im2col(x, k, k, 2, pad), ws[0])
    mag = orc.bf16_gemm(np.abs(orc.im2col(x, k, k, 2, pad)), np.abs(ws[0]))
    assert np.all(np.abs(host(ys[0]) - orc.activation(ref, act)) <= k * k * c * 2.0 ** -23 * mag + 1e-30)
    only = [None, torch.full_like(ys[1], float("nan")), torch.full_like(ys[2], float("nan"))]
    model.eval_config(bits, xd, batch, only)
    ctx.check_sync()
    assert torch.equal(only[1], ys[1]) and torch.equal(only[2], ys[2])
    ctx.set_prefix_reuse(True)
    try:
        for b2 in ([16, 8, 5], [16, 4, 5], [16, 4, 8], [16, 8, 5]):       # a changed reader brings the pooled input back
            model.eval_config(b2, xd, batch, only)
        ctx.check_sync()
        assert torch.equal(only[1], ys[1]) and torch.equal(only[2], ys[2])
    finally:
        ctx.set_prefix_reuse(False)
    model.close()


def _conv_both_ways(ctx, c, n, h, wd, pad, batch, widths=((8, 8, 8), (8, 5, 4))):
    """A stride-1 3x3 convolution between a 1x1 layer and a reader of its codes: codes and output with implicit convolutions
    are those of the patch matrix, bit for bit.  Returns the forms of the implicit runs' launches."""
    L = wl.Layer
    oh, ow = h + 2 * pad - 2, wd + 2 * pad - 2
    layers = [L("in", c, 16, src=-1, kh=1, kw=1, stride=1, in_h=h, in_w=wd, in_c=16, src_h=h, src_w=wd),
              L("conv", n, 9 * c, src=0, act=orc.ACT_RELU, kh=3, kw=3, stride=1, pad=pad, in_h=h, in_w=wd, in_c=c, src_h=h, src_w=wd),
              L("out", 16, n, src=1, kh=1, kw=1, stride=1, in_h=oh, in_w=ow, in_c=n, src_h=oh, src_w=ow)]
    rng = np.random.default_rng(c + n + h)
    x = rng.standard_normal((batch, h, wd, 16)).astype(np.float32)
    ws = [(rng.standard_normal((l.n_out, l.k_in)) / np.sqrt(l.k_in)).astype(np.float32) for l in layers]
    model, xd = build(ctx, wl.Workload("conv", 1, layers, batch, x, ws))
    rows = batch * oh * ow
    forms = []
    try:
        for bits in widths:
            got = []
            for implicit in (True, False):
                ctx.set_implicit_conv(implicit)
                y = torch.full((rows, 16), float("nan"), device="cuda")
                before = ctx.launch_forms()
                model.eval_config(list(bits), xd, batch, [None, None, y])
                if implicit:
                    forms += [f for f, v in ctx.launch_forms().items() if f.startswith("conv") for _ in range(v - before[f])]
                qx = torch.zeros((rows, n), dtype=torch.int8, device="cuda")
                model.debug_dump(2, qx, None, None)
                ctx.check_sync()
                got.append((qx, y))
            assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])
            assert got[0][0].any()
    finally:
        ctx.set_implicit_conv(True)
    model.close()
    return forms


@pytest.mark.parametrize("c,n,h,wd,pad,batch,form", [
    (64, 64, 56, 56, 1, 4, "slab"), (64, 64, 9, 9, 1, 80, "slab"), (64, 32, 11, 7, 1, 90, "slab"), (128, 128, 28, 28, 1, 13, "slab"),
    (128, 96, 5, 5, 2, 230, "slab"), (64, 64, 130, 6, 1, 13, "slab"), (64, 32, 8, 8, 0, 160, "slab"), (256, 256, 14, 14, 1, 128, "streamed"),
    (256, 256, 14, 14, 1, 77, "im2col"), (512, 512, 7, 7, 1, 129, "streamed"), (192, 288, 13, 17, 0, 30, "streamed"), (64, 320, 6, 140, 1, 8, "streamed"),
    (128, 160, 28, 28, 1, 11, "streamed"), (64, 256, 64, 64, 1, 5, "streamed"), (256, 224, 14, 14, 2, 70, "streamed"), (128, 128, 28, 28, 1, 2, "im2col"),
    (64, 64, 20, 20, 3, 20, "slab"), (128, 256, 20, 20, 3, 20, "streamed"), (64, 96, 12, 30, 5, 20, "slab")])
def test_convolution_by_slabs_matches_the_patch_matrix(ctx, c, n, h, wd, pad, batch, form):
    """Stride-1 3x3 convolutions whose only output is their reader's int8 codes load their input once per tile.  Tiles that
    are whole rows, parts of rows and whole images, halos shared and not, padding up to and beyond what a tap reaches, 64- and
    128-byte chunks, weights resident and streamed, one and several column tiles, CTA pairs with an odd last tile; few tiles
    stay with the other kernel: the form it names (on 148 SMs), codes bit for bit."""
    assert _conv_both_ways(ctx, c, n, h, wd, pad, batch) == ["conv_" + form] * 2


@pytest.mark.parametrize("c,n,h,wd,batch", [(256, 256, 14, 14, 128), (128, 256, 28, 28, 20), (128, 128, 28, 28, 13)])
def test_convolution_by_slabs_without_cta_pairs(ctx, c, n, h, wd, batch):
    """128-byte chunks with one CTA per tile, weights streamed and resident."""
    ctx.set_pair_tiles(False)
    try:
        assert _conv_both_ways(ctx, c, n, h, wd, 1, batch) == ["conv_streamed" if n > 128 else "conv_slab"] * 2
    finally:
        ctx.set_pair_tiles(True)


def test_stem_writes_the_codes_of_its_pooled_readers(ctx):
    """Five readers of a pooled stem on four grids, one of them 16 bit: two int8 grids leave with the pooled tensor, the
    others quantize for themselves; outputs and codes are those of a run in which every reader does.  Then one reader's
    width at a time changes under prefix reuse."""
    L = wl.Layer
    h, wd, batch, n = 37, 62, 3, 48
    oh, ow = (h - 1) // 2 + 1, (wd - 1) // 2 + 1
    ph, pw = (oh - 1) // 2 + 1, (ow - 1) // 2 + 1
    reader = dict(src=0, kh=1, kw=1, stride=1, in_h=ph, in_w=pw, in_c=n, pool_before=wl.POOL_MAX3S2, src_h=oh, src_w=ow)
    layers = [L("stem", n, 147, src=-1, act=orc.ACT_RELU, kh=7, kw=7, stride=2, pad=3, in_h=h, in_w=wd, in_c=3, src_h=h, src_w=wd)]
    layers += [L(f"r{i}", 16 + 8 * i, n, **reader) for i in range(5)]
    rng = np.random.default_rng(11)
    x = rng.standard_normal((batch, h, wd, 3)).astype(np.float32)
    ws = [(rng.standard_normal((l.n_out, l.k_in)) / np.sqrt(l.k_in)).astype(np.float32) for l in layers]
    model, xd = build(ctx, wl.Workload("stem", 1, layers, batch, x, ws))
    rows = batch * ph * pw

    def run(bits):
        ys = [None] + [torch.full((rows, l.n_out), float("nan"), device="cuda") for l in layers[1:]]
        model.eval_config(bits, xd, batch, ys)
        codes = []
        for l in range(1, 6):
            q = torch.zeros((rows, n), dtype=torch.int8, device="cuda")
            if bits[l] != 16:
                model.debug_dump(l, q, None, None)
            codes.append(q)
        ctx.check_sync()
        return ys[1:] + codes

    want = {}
    steps = ([16, 8, 5, 16, 3, 8], [16, 8, 5, 16, 3, 4], [16, 6, 5, 16, 3, 4], [16, 6, 5, 8, 3, 4], [16, 8, 5, 16, 3, 8])
    try:
        ctx.set_fusion(False)
        for bits in steps:
            want[tuple(bits)] = run(bits)
        ctx.set_fusion(True)
        for reuse in (False, True):
            ctx.set_prefix_reuse(reuse)
            for bits in steps:
                for a, b in zip(run(bits), want[tuple(bits)]):
                    assert torch.equal(a, b)
    finally:
        ctx.set_fusion(True)
        ctx.set_prefix_reuse(False)
    model.close()


@pytest.mark.parametrize("m,k,off", [(33, 75, 0), (400, 96, 1), (5, 1030, 0)])
def test_operands_on_several_grids_come_from_one_pass(ctx, m, k, off):
    """Six layers on five grids (more than one pass writes) that read the same rows of the external input, next to one that
    reads other columns: codes, accumulators and outputs against the oracle, rows on and off 16 bytes."""
    import paper_2302_01382_b200 as q
    L = wl.Layer
    layers = [L(f"l{i}", 24 + i, k, src=-1) for i in range(6)] + [L("slice", 16, 32, src=-1, src_col0=16)]
    rng = np.random.default_rng(m + k)
    ws = [(rng.standard_normal((l.n_out, l.k_in)) / np.sqrt(l.k_in)).astype(np.float32) for l in layers]
    w = wl.Workload("grids", 1, layers, m, rng.standard_normal((m, k)).astype(np.float32), ws)
    model = q.Model(ctx, layers, [dev(a) for a in ws])
    buf = torch.zeros(m * k + 4, device="cuda")
    x = buf[off:off + m * k].reshape(m, k)
    x.copy_(dev(w.x))
    model.calibrate_model(x, m)
    act_g, w_amax = check_calibration(model, w)
    for bits in ([8, 4, 16, 4, 5, 3, 8], [16, 16, 8, 2, 8, 6, 16]):
        ys = run_eval(ctx, model, w, x, bits)
        teacher_forced_check(ctx, model, w, x, bits, ys, act_g, w_amax)
    model.close()


def test_readers_of_one_source_in_two_geometries_have_operands_of_their_own(ctx):
    """Two pooling readers that declare one source with transposed sizes: each pools it as it says, at equal and at different
    widths, and a size that is not the source's is refused whatever the widths of its neighbours."""
    import paper_2302_01382_b200 as q
    L = wl.Layer
    reader = dict(src=0, kh=1, kw=1, stride=1, in_h=5, in_w=7, in_c=32, pool_before=wl.POOL_MAX3S2)
    layers = [L("in", 32, 16, src=-1, kh=1, kw=1, stride=1, in_h=10, in_w=14, in_c=16, src_h=10, src_w=14),
              L("a", 24, 32, src_h=10, src_w=14, **reader), L("b", 20, 32, src_h=14, src_w=10, **reader),
              L("c", 16, 32, src_h=14, src_w=10, **reader)]
    rng = np.random.default_rng(7)
    x = rng.standard_normal((3, 10, 14, 16)).astype(np.float32)
    ws = [(rng.standard_normal((l.n_out, l.k_in)) / np.sqrt(l.k_in)).astype(np.float32) for l in layers]
    w = wl.Workload("geometries", 1, layers, 3, x, ws)
    model, xd = build(ctx, w)
    act_g, w_amax = check_calibration(model, w)
    for bits in ([8, 8, 8, 8], [8, 8, 4, 4], [8, 4, 8, 6], [16, 16, 8, 8], [8, 8, 16, 16]):
        teacher_forced_check(ctx, model, w, xd, bits, run_eval(ctx, model, w, xd, bits), act_g, w_amax)
    model.close()
    for i in (1, 2, 3):
        bad = [L(**{**vars(l), "src_w": l.src_w + 1}) if j == i else l for j, l in enumerate(layers)]
        model = q.Model(ctx, bad, [dev(a) for a in ws])
        with pytest.raises(q.QcfgError) as e:
            model.calibrate_model(xd, 3)
        assert e.value.status == q.ESHAPE
        model.close()


@pytest.mark.parametrize("c,n,h,wd,batch,form", [
    (128, 128, 40, 40, 8, "conv_im2col"), (128, 96, 40, 40, 8, "conv_im2col"), (128, 64, 40, 40, 8, "conv_slab"), (64, 128, 40, 40, 8, "conv_slab"),
    (128, 128, 44, 44, 8, "conv_slab")])
def test_slab_weights_of_one_column_tile_are_resident(ctx, c, n, h, wd, batch, form):
    """A convolution of up to 128 columns goes by slabs only where its weights fit beside them: 40 x 40 x 128 is cut into slabs
    of 27 KB, three of which leave no room for 144 KB of weights."""
    assert _conv_both_ways(ctx, c, n, h, wd, 1, batch) == [form] * 2
