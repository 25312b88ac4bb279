"""The ends of FP32's range in the general forward kernel: densities below
2^-126, the smallest normal number, and infinite weights, inputs and hidden
values, which the operands of FP32 inference do not hold, against the CUDA-core
kernel that does."""
import math

import numpy as np
import pytest

import mixtures
import oracle
import synth
from gpu_helpers import cuda, host, make_model

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

NET = synth.Workload(name="one level of 4 features, 4-32-16", mode=synth.RADIANCE, level_res=[8], feat=4,
                     log2_table=12, widths=[4, 32, 16], K=4)


@pytest.fixture(autouse=True)
def _need_cuda():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")


@pytest.mark.parametrize("precision,bar", [(synth.FP32, 1e-4), (synth.FP32_TC, 1e-4), (synth.BF16X3, 2e-2)],
                         ids=["fp32", "fp32tc", "bf16x3"])
def test_densities_below_the_normal_range(precision, bar):
    # Four sharp lobes of one mean, seen from around its opposite: densities
    # of 3e-39 to 4e-38. A lobe's term is held to a unit of 2^-149 before the
    # factor of up to 7.4 that normalises it, hence 4 x 8 units beside the bar.
    lobes = dict(lams=[0.4, 0.3, 0.2, 0.1], kaps=[45.0, 45.5, 46.0, 46.5], thetas=[0.7] * 4, phis=[1.0] * 4)
    w = NET.with_(precision=precision)
    params = mixtures.diverse_params(w, mixtures.raw_for(**lobes), mixtures.X0).astype(np.float32)
    n = 512
    pos = np.repeat(np.array(mixtures.X0, np.float32)[:, None], n, axis=1)
    th, ph = math.pi - 0.7 + 0.3 * np.linspace(-1, 1, n), math.pi + 1.0 + 0.3 * np.cos(np.arange(n))
    dirs = np.stack([np.sin(th) * np.cos(ph), np.sin(th) * np.sin(ph), np.cos(th)]).astype(np.float32)
    ref = oracle.eval_pdf64(w, params, pos, dirs.astype(np.float64))
    assert ref.min() < 2.0 ** -126 < ref.max()
    m = make_model(w, params, n, precision=precision)
    v = host(m.eval_pdf(cuda(pos), cuda(dirs))).astype(np.float64)
    m.check_device_status()
    assert np.all(np.abs(v - ref) <= bar * ref + 32 * 2.0 ** -149)


# Networks of every instance of the FP32 forward: two features a level, four,
# others (an odd number of inputs before the product-mode ones), sixteen lobes.
NETS = [synth.Workload(name="two features", mode=synth.RADIANCE, level_res=[4, 7, 12, 40], feat=2, log2_table=12,
                       widths=[8, 64, 32, 32], K=8),
        synth.Workload(name="four features", mode=synth.RADIANCE, level_res=[6, 30], feat=4, log2_table=13,
                       widths=[8, 32, 16], K=4),
        synth.Workload(name="four features, 128 wide", mode=synth.RADIANCE, level_res=[6, 30], feat=4,
                       log2_table=13, widths=[8, 128, 64, 16], K=4),
        synth.Workload(name="one feature, product", mode=synth.PRODUCT, level_res=[5, 9, 30], feat=1, log2_table=12,
                       widths=[24, 16, 8], K=2),
        synth.Workload(name="sixteen lobes", mode=synth.PRODUCT, level_res=[6, 11, 40], feat=2, log2_table=12,
                       widths=[28, 64, 64], K=16)]


def _queries(w, n):
    uu = synth.uniform_rows(71, synth.S_DIR, 2, n)
    aux = synth.aux_inputs(71, n) if w.mode == synth.PRODUCT else None
    return synth.positions(71, n), synth.sphere_dirs(uu[0], uu[1]).astype(np.float32), aux


def _both(w, params, pos, dirs, aux):
    """Densities of the model's FP32 inference (three BF16 parts) and of the
    CUDA-core kernel, which computes in FP32 throughout."""
    import ctypes as C

    import paper_2504_04315_gb300 as npm
    from paper_2504_04315_gb300 import _lib
    n = pos.shape[1]
    p, d, a = cuda(pos), cuda(dirs), None if aux is None else cuda(aux)
    m = make_model(w, params, n, precision=synth.FP32)
    got = host(m.eval_pdf(p, d, a))
    m.check_device_status()
    cfg, theta, out = npm.config_from(w, max_batch=n, precision=synth.FP32), cuda(params), torch.empty(n, device="cuda")
    _lib.check(_lib.load().npm_eval_pdf_noalloc(
        C.byref(cfg), theta.data_ptr(), n, p.data_ptr(), None if a is None else a.data_ptr(), d.data_ptr(), n,
        out.data_ptr(), torch.cuda.current_stream().cuda_stream), "npm_eval_pdf_noalloc")
    return got, host(out)


def _layers(w):
    o = sum(synth.grid_sizes(w)) * w.feat
    for a, b in zip(w.widths[:-1], w.widths[1:]):
        yield o, a, b
        o += a * b


@pytest.mark.parametrize("value", [np.inf, -np.inf])
@pytest.mark.parametrize("w", NETS, ids=lambda w: w.name)
def test_an_infinite_weight_shows(w, value):
    pos, dirs, aux = _queries(w, 700)
    shown = 0
    for o, a, b in _layers(w):
        params = synth.random_params(w, 72)
        params[o + (b // 2) * a + 1] = value
        got, want = _both(w, params, pos, dirs, aux)
        shown += np.isnan(want).sum()
        assert np.isnan(got[np.isnan(want)]).all(), (o, np.isnan(got).sum(), np.isnan(want).sum())
    assert shown >= 350


@pytest.mark.parametrize("w", NETS, ids=lambda w: w.name)
def test_infinite_inputs_and_hidden_values_show(w):
    n = 700
    pos, dirs, aux = _queries(w, n)
    params = synth.random_params(w, 73)
    layers = list(_layers(w))
    # An infinite feature at the box's low corner, where the first half lies;
    # the second half lies away from it.
    pos[:, :n // 2] = 0.0
    pos[:, n // 2:] = 0.5 + 0.5 * pos[:, n // 2:]
    grid = params.copy()
    grid[0] = np.inf
    cases = [(grid, aux)]
    if aux is not None:
        rough = aux.copy()
        rough[6, :n // 2] = np.inf
        cases.append((params, rough))
    for p, a in cases:
        got, want = _both(w, p, pos, dirs, a)
        # (the CUDA-core kernel's ReLU takes infinity less infinity for zero)
        assert np.isnan(got[:n // 2]).all() and np.isnan(got[np.isnan(want)]).all()
        rest = got[n // 2:], want[n // 2:]
        assert np.all(np.abs(rest[0] - rest[1]) <= 1e-4 * rest[1])
    # Hidden values of the last hidden layer that overflow, for some queries
    # (sums of values of one sign, which overflow in any order).
    o, a, b = layers[-2]
    big = params.copy()
    big[:layers[0][0]] = 8.0 * np.abs(big[:layers[0][0]])
    wl = np.abs(big[o:o + a * b].reshape(b, a)) * np.float32(2.0 ** 127.5)
    if len(layers) == 2:
        wl[:, len(w.level_res) * w.feat:] = 0.0  # (the product-mode inputs come with both signs)
    big[o:o + a * b] = wl.ravel()
    big[layers[-1][0]:] *= np.float32(2.0 ** -60)  # (finite ones leave finite outputs)
    assert np.isfinite(big).all()
    got, want = _both(w, big, pos, dirs, aux)
    assert np.isnan(want).any() and np.isnan(got[np.isnan(want)]).all()


@pytest.mark.parametrize("w", NETS, ids=lambda w: w.name)
def test_finite_values_and_nan_stay_as_in_fp32(w):
    pos, dirs, aux = _queries(w, 700)
    # ReLU takes a NaN weight of a hidden layer for zero.
    params = synth.random_params(w, 74)
    o, a, b = list(_layers(w))[-2]
    params[o + 3 * a + 2] = np.nan
    got, want = _both(w, params, pos, dirs, aux)
    assert np.isfinite(want).all() and np.all(np.abs(got - want) <= 1e-4 * want)
    # A hidden value between BF16's and FP32's largest is not an infinite one.
    params = synth.random_params(w, 75)
    ng = sum(synth.grid_sizes(w)) * w.feat
    params[:ng] = 1.0
    for o, a, b in _layers(w):
        params[o:o + a * b] = 0.0
    for i, (o, a, b) in enumerate(_layers(w)):
        params[o] = 3.395e38 if i == 0 else 1e-38 if i == len(w.widths) - 2 else 1.0
    got, want = _both(w, params, pos, dirs, aux)
    assert np.isfinite(want).all() and np.isfinite(got).all()


# (70,000 queries: more tiles than three groups on every SM hold, fewer than
# four, which takes the two-feature instance of four.)
@pytest.mark.parametrize("n", [700, 70000])
@pytest.mark.parametrize("w", NETS, ids=lambda w: w.name)
def test_nan_inputs_stay_as_in_fp32(w, n):
    # ReLU takes the first layer's outputs for a NaN input for zero: the
    # density is that of raw outputs of zero.
    pos, dirs, aux = _queries(w, n)
    params = synth.random_params(w, 76)
    params[1] = np.nan  # a feature at the box's low corner
    pos[:, :n // 3] = 0.0
    if aux is not None:
        aux[4, n // 3:n // 2] = np.nan
    got, want = _both(w, params, pos, dirs, aux)
    assert np.isfinite(want).all() and np.all(np.abs(got - want) <= 1e-4 * want)
