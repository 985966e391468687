"""E_N (Eqs. 3-5) through the C-ABI against the noise oracle."""
import numpy as np
import pytest
import torch

import qcfg_workloads as wl
from oracle import noise_oracle as nz

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import paper_2302_01382_b200 as q
    c = q.Context(0)
    yield c
    c.close()


def _run(ctx, w, nus, lam):
    import paper_2302_01382_b200 as q
    weights = [torch.from_numpy(a).cuda() for a in w.weights]
    model = q.Model(ctx, w.layers, weights)
    x = torch.from_numpy(np.ascontiguousarray(w.x)).cuda()
    noises = [None if a is None else torch.from_numpy(a).cuda() for a in nus]
    e = model.noise_sensitivity(x, w.m, noises, lam)
    ctx.check_sync()
    model.close()
    return np.array(e)


def _ragged_mlp(sizes, m):
    """Rows that are no whole groups of four or eight elements, outputs that are no multiple of four."""
    rng = np.random.default_rng(sum(sizes))
    layers = wl.mlp_layers(sizes)
    ws = [(rng.standard_normal((l.n_out, l.k_in)) / np.sqrt(l.k_in)).astype(np.float32) for l in layers]
    return wl.Workload("ragged", 1, layers, m, rng.standard_normal((m, sizes[0])).astype(np.float32), ws)


@pytest.mark.parametrize("make", [lambda: wl.tiny_mlp(), lambda: _ragged_mlp((37, 1030, 22, 7), 33), lambda: _ragged_mlp((2052, 1500, 9, 3), 5),
                                  lambda: wl.bert_stack(41, 333, 128, 512, 2),
                                  lambda: wl.resnet50(seed=3, batch=2, in_hw=32, width=16, n_classes=10, blocks=(1, 1, 1, 1))])
def test_noise_sensitivity_matches_oracle(ctx, make):
    w = make()
    nus = wl.standard_normal_like(w.weights, 99)
    nus[1] = None                                         # a skipped layer reports 0
    lam = 0.05
    got = _run(ctx, w, nus, lam)
    want = np.array(nz.noise_sensitivity(w.layers, w.weights, w.x, nus, lam))
    assert got[1] == 0.0 and want[1] == 0.0
    # both sides round operands to bf16; the GPU accumulates in fp32, the oracle wider, so a few
    # intermediate activations round to the other bf16 neighbour: agreement to about 1e-3 of E_N,
    # 1e-2 required, with a floor for layers whose effect is below the rounding noise
    np.testing.assert_allclose(got, want, rtol=1e-2, atol=2e-4)
    # layers nothing downstream reads: exactly zero on both sides
    assert np.array_equal(got == 0.0, want == 0.0)
    # and the ordering of clearly separated layers (the use the paper makes of the metric) agrees
    order = np.argsort(want)
    for a, b in zip(order[:-1], order[1:]):
        if want[b] > 1.05 * want[a] + 4e-4:
            assert got[b] > got[a]


def test_noise_sensitivity_runs_only_what_a_perturbation_reaches(ctx):
    """Parallel branches: the layers an earlier perturbation reached and the next one does not are run again, so
    every E_N equals that of a call which perturbs this layer alone, bit for bit; with the switch for reuse
    between calls on, a changed input gives the changed input's result."""
    w = wl.resnet50(seed=8, batch=2, in_hw=32, width=16, n_classes=10, blocks=(2, 1, 1, 1))
    nus = wl.standard_normal_like(w.weights, 5)
    both = _run(ctx, w, nus, 0.05)
    for l in (1, 2, 3, 4, 7, len(nus) - 1):
        alone = _run(ctx, w, [n if i == l else None for i, n in enumerate(nus)], 0.05)
        assert alone[l] == both[l] and np.count_nonzero(alone) <= 1
    ctx.set_prefix_reuse(True)
    try:
        assert np.array_equal(_run(ctx, w, nus, 0.05), both)
    finally:
        ctx.set_prefix_reuse(False)


def test_noise_sensitivity_zero_lambda_and_errors(ctx):
    import paper_2302_01382_b200 as q
    w = wl.tiny_mlp()
    nus = wl.standard_normal_like(w.weights, 3)
    assert np.all(_run(ctx, w, nus, 0.0) == 0.0)
    weights = [torch.from_numpy(a).cuda() for a in w.weights]
    model = q.Model(ctx, w.layers, weights)
    x = torch.from_numpy(w.x).cuda()
    with pytest.raises(q.QcfgError) as e:
        model.noise_sensitivity(x, w.m, [None] * 3, -1.0)
    assert e.value.status == q.EINVAL
    model.close()


@pytest.mark.parametrize("k,cols", [(37, 19), (64, 32)])
def test_noise_beyond_the_range_of_32_bits(ctx, k, cols):
    """A deviation that overflows makes every perturbed weight infinite and nothing else: with positive weights, inputs and
    draws the output is infinite, not NaN, which a deviation that reached the zeros behind a row's last column would give."""
    rng = np.random.default_rng(k)
    layers = wl.mlp_layers((k, cols))
    ws = [rng.uniform(0.5, 1.5, (l.n_out, l.k_in)).astype(np.float32) for l in layers]
    w = wl.Workload("range", 1, layers, 33, rng.uniform(0.5, 1.5, (33, k)).astype(np.float32), ws)
    nus = [rng.uniform(1.0, 2.0, a.shape).astype(np.float32) for a in ws]
    assert np.isfinite(_run(ctx, w, nus, 1.0)).all()
    assert np.isposinf(_run(ctx, w, nus, 3.4e38)).all()


@pytest.mark.parametrize("value", [np.inf, np.nan])
def test_non_finite_weight_reaches_every_row_through_the_deviation(ctx, value):
    """The tensor's maximum is folded from the rows' maxima as an integer, where an infinity or a NaN in one row wins: with draws
    of zero every perturbed weight of the layer is NaN.  ReLU turns its outputs into zeros, so the last output is zero and its
    distance is exactly 1, unless the unperturbed output is infinite itself."""
    w = _ragged_mlp((37, 1030, 22, 7), 33)
    w.weights[1][20, 1029] = value
    nus = [np.zeros_like(a) for a in w.weights]
    nus[0] = nus[2] = None
    e = _run(ctx, w, nus, 0.05)
    assert e[0] == 0.0 and e[2] == 0.0
    assert e[1] == 1.0 if np.isnan(value) else not np.isfinite(e[1])
