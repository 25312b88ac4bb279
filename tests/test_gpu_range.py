"""The ends of FP32's range in the general forward kernel: densities below
2^-126, the smallest normal number."""
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
