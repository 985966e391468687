"""Prefix reuse between consecutive configurations (the searches change one layer, or a slice of
the ordering, per evaluation): with reuse on, every evaluation of a search sequence must give
bit-identical outputs to a full recompute, while launching fewer kernels."""
import numpy as np
import pytest
import torch

import qcfg_workloads as wl

pytestmark = pytest.mark.gpu


def _sequences(n, rng):
    order = [int(i) for i in rng.permutation(n)]
    accept = rng.random(n) < 0.5
    greedy = wl.greedy_sequence(order, accept)
    bisect = wl.bisection_sequence(order, rng.random(8) < 0.5, max(2, (3 * n) // 4), 8)
    wild = [rng.choice(np.array([4, 8, 16], np.uint8), size=n) for _ in range(6)]
    return greedy[:24] + bisect + wild + [wild[-1], wild[-1]]      # the last two: nothing changes


@pytest.mark.parametrize("kind", ["bert", "bert_wide_qkv", "resnet"])
def test_reuse_is_bit_identical_on_search_sequences(kind):
    import paper_2302_01382_b200 as q
    rng = np.random.default_rng(11)
    if kind == "bert":
        w = wl.bert_stack(21, 640, 256, 1024, 3, bit_choices=None)
    elif kind == "bert_wide_qkv":
        w = wl.bert_stack_wide_qkv(22, 384, 256, 1024, 2)
    else:
        w = wl.resnet50(seed=23, batch=2, in_hw=64, width=16, n_classes=24, blocks=(2, 1, 1, 1))
    n = len(w.layers)
    ctx = q.Context(0)
    try:
        weights = [torch.from_numpy(a).cuda() for a in w.weights]
        x = torch.from_numpy(w.x).cuda()
        model = q.Model(ctx, w.layers, weights)
        model.calibrate_model(x, w.m)
        rows_out = wl.layer_rows(w.layers, n - 1, w.m)
        out_a = torch.empty((rows_out, w.layers[-1].n_out), device="cuda")
        out_b = torch.empty_like(out_a)
        tap = n // 2
        tap_a = torch.empty((wl.layer_rows(w.layers, tap, w.m), w.layers[tap].n_out), device="cuda")
        tap_b = torch.empty_like(tap_a)
        seq = _sequences(n, rng)
        # reference: full recompute of every configuration
        ref, launches_full = [], 0
        for i, bits in enumerate(seq):
            ys = [None] * n
            ys[-1] = out_a
            if i % 5 == 3:
                ys[tap] = tap_a
            l0 = ctx.launch_count()
            model.eval_config(bits, x, w.m, ys)
            launches_full += ctx.launch_count() - l0
            ctx.check_sync()
            ref.append((out_a.clone(), tap_a.clone() if i % 5 == 3 else None))
        ctx.set_prefix_reuse(True)
        launches_reuse = 0
        for i, bits in enumerate(seq):
            ys = [None] * n
            ys[-1] = out_b
            if i % 5 == 3:
                ys[tap] = tap_b
            l0 = ctx.launch_count()
            model.eval_config(bits, x, w.m, ys)
            launches_reuse += ctx.launch_count() - l0
            ctx.check_sync()
            assert torch.equal(out_b, ref[i][0]), f"{kind}: configuration {i} differs under reuse"
            if ref[i][1] is not None:
                assert torch.equal(tap_b, ref[i][1]), f"{kind}: tapped layer differs at configuration {i}"
        assert launches_reuse < launches_full
        # a switch in between invalidates what is kept: the next evaluation is a full one and still right
        ctx.set_fusion(False)
        ys = [None] * n
        ys[-1] = out_b
        model.eval_config(seq[3], x, w.m, ys)
        ctx.check_sync()
        assert torch.equal(out_b, ref[3][0])
        model.close()
    finally:
        ctx.close()


def _taps(model, w, bits):
    """Operand codes and accumulators of every integer layer after the last evaluation."""
    out = []
    for l, layer in enumerate(w.layers):
        if bits[l] == 16:
            out.append(None)
            continue
        rows = wl.layer_rows(w.layers, l, w.m)
        qx = torch.empty((rows, layer.k_in), dtype=torch.int8, device="cuda")
        acc = torch.empty((rows, layer.n_out), dtype=torch.int32, device="cuda")
        model.debug_dump(l, qx, None, acc)
        out.append((qx, acc))
    return out


@pytest.mark.parametrize("kind", ["fan", "bert", "bert_wide_qkv", "resnet"])
def test_taps_after_partial_forwards(kind):
    """debug_dump reads what every layer ran with, also where the last evaluation skipped the layer and layers
    that shared its codes have changed their width since: under prefix reuse and after a search."""
    import paper_2302_01382_b200 as q
    rng = np.random.default_rng(12)
    if kind == "fan":            # layers on one input, which share one operand at equal widths
        w = wl.bert_stack(24, 300, 128, 512, 1, bit_choices=None)
    elif kind == "bert":
        w = wl.bert_stack(21, 200, 128, 512, 3, bit_choices=None)
    elif kind == "bert_wide_qkv":
        w = wl.bert_stack_wide_qkv(22, 200, 128, 512, 2)
    else:
        w = wl.resnet50(seed=23, batch=2, in_hw=64, width=16, n_classes=24, blocks=(2, 1, 1, 1))
    n = len(w.layers)
    ctx, full = q.Context(0), q.Context(0)
    try:
        weights = [torch.from_numpy(a).cuda() for a in w.weights]
        x = torch.from_numpy(w.x).cuda()
        model, plain = q.Model(ctx, w.layers, weights), q.Model(full, w.layers, weights)
        for mod in (model, plain):
            mod.calibrate_model(x, w.m)
        y = torch.empty((wl.layer_rows(w.layers, n - 1, w.m), w.layers[-1].n_out), device="cuda")
        ys = [None] * (n - 1) + [y]

        def same_taps(bits, what):
            plain.eval_config(bits, x, w.m, ys)
            for l, (got, want) in enumerate(zip(_taps(model, w, bits), _taps(plain, w, bits))):
                if want is not None:
                    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1]), f"{kind}, {what}: tap of layer {l}"

        if kind == "fan":
            seq = [[8] * n, [4] + [8] * (n - 1), [4, 4] + [8] * (n - 2), [8, 4] + [8] * (n - 2), [16, 4, 2] + [8] * (n - 3), [8] * n]
        else:
            seq = [list(map(int, b)) for b in _sequences(n, rng)[::4]]
        ctx.set_prefix_reuse(True)
        for i, bits in enumerate(seq):
            model.eval_config(bits, x, w.m, ys)
            same_taps(bits, f"configuration {i}")
        ctx.set_prefix_reuse(False)
        for algorithm in (0, 1):
            order = [int(i) for i in rng.permutation(n)]
            _, visited, _, n_evals = model.search(algorithm, order, [8, 4], 0.9, x, w.m)
            assert n_evals > 0
            same_taps(list(visited[-1]), f"search {algorithm}")
        ctx.check_sync()
        full.check_sync()
        model.close()
        plain.close()
    finally:
        ctx.close()
        full.close()


def test_a_changed_reader_of_a_pooled_stem_does_not_run_the_stem_again():
    """Under reuse a layer that reads the max-pooled stem goes on from the pooled tensor: one launch builds its operand and
    one multiplies it.  A change of the stem itself runs everything again."""
    import paper_2302_01382_b200 as q
    L = wl.Layer
    layers = [L("stem", 32, 147, src=-1, act=wl.ACT_RELU, kh=7, kw=7, stride=2, pad=3, in_h=32, in_w=32, in_c=3, src_h=32, src_w=32)]
    for name, n in (("a", 24), ("b", 16)):
        layers.append(L(name, n, 32, src=0, kh=1, kw=1, stride=1, in_h=8, in_w=8, in_c=32, pool_before=wl.POOL_MAX3S2, src_h=16, src_w=16))
    g = torch.Generator(device="cuda").manual_seed(3)
    weights = [torch.randn((l.n_out, l.k_in), generator=g, device="cuda") for l in layers]
    x = torch.randn((5, 32, 32, 3), generator=g, device="cuda")
    ctx, full = q.Context(0), q.Context(0)
    try:
        model, plain = q.Model(ctx, layers, weights), q.Model(full, layers, weights)
        ys = [None] + [torch.empty((5 * 64, n), device="cuda") for n in (24, 16)]
        want = [None] + [torch.empty_like(y) for y in ys[1:]]
        for mod in (model, plain):
            mod.calibrate_model(x, 5)
        ctx.set_prefix_reuse(True)
        for bits, changed in (([16, 8, 5], 0), ([16, 4, 5], 0), ([16, 4, 8], 0), ([16, 8, 8], 1), ([16, 8, 5], 2), ([8, 8, 5], 0),
                              ([16, 8, 5], 0), ([16, 4, 5], 1)):
            before = ctx.launch_count()
            model.eval_config(bits, x, 5, [y if changed in (0, i) else None for i, y in enumerate(ys)])
            launches = ctx.launch_count() - before
            if changed:
                assert launches == 2, (bits, launches)
            plain.eval_config(bits, x, 5, want)
            ctx.check_sync()
            full.check_sync()
            for i in (1, 2):
                if changed in (0, i):
                    assert torch.equal(ys[i], want[i]), (bits, i)
        model.close()
        plain.close()
    finally:
        ctx.close()
        full.close()
