"""The tensor-core forward kernel at the edges of its tiles and groups: one
query, a tile less or more one, one tile per SM, as many as four tile groups
per SM hold and one query more, on networks whose inputs fill the activation columns unevenly
(an odd number of one-feature levels before the product-mode inputs, an odd
number of two-feature levels, three-feature levels, 128-wide layers, sixteen
lobes). Densities at the sampled directions against the FP64 oracle: 1e-4 in
FP32 and the FP32-accuracy mode, 2e-2 at the 99.9th percentile (the
reduced-precision bar, denominator floored at 1e-2 / (4 pi)) otherwise."""
import math

import numpy as np
import pytest

import oracle
import synth
from gpu_helpers import cuda, host, make_model

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

ODD_ONE = synth.Workload(name="3 levels x 1 feat, product", mode=synth.PRODUCT, level_res=[5, 9, 30], feat=1,
                         log2_table=12, widths=[24, 16, 8], K=2)
ODD_TWO = synth.Workload(name="5 levels x 2 feats", mode=synth.RADIANCE, level_res=[4, 7, 12, 25, 40], feat=2,
                         log2_table=13, widths=[12, 32, 32], K=8)
LOBES16 = synth.Workload(name="3 levels x 2 feats, product, K=16", mode=synth.PRODUCT, level_res=[6, 11, 40], feat=2,
                         log2_table=12, widths=[28, 64, 64], K=16)
WIDE = synth.Workload(name="2 levels x 4 feats, 128 wide", mode=synth.RADIANCE, level_res=[6, 30], feat=4,
                      log2_table=13, widths=[8, 128, 20], K=5)
WIDE_TWO = synth.Workload(name="2 levels x 2 feats, 96 wide", mode=synth.RADIANCE, level_res=[6, 30], feat=2,
                          log2_table=13, widths=[4, 96, 20], K=5)

THREE = synth.Workload(name="3 levels x 3 feats", mode=synth.RADIANCE, level_res=[6, 11, 40], feat=3,
                       log2_table=12, widths=[12, 32, 12], K=3)

PRECISIONS = {"fp32": synth.FP32, "fp32tc": synth.FP32_TC, "bf16x3": synth.BF16X3, "fp16": synth.FP16}
# Three features per level are FP32's alone.
CASES = [(w, p) for w in (ODD_ONE, ODD_TWO, LOBES16, WIDE, WIDE_TWO) for p in PRECISIONS] + [(THREE, "fp32")]


@pytest.fixture(autouse=True)
def _need_cuda():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")


@pytest.mark.parametrize("w,precision", CASES, ids=lambda v: v if isinstance(v, str) else v.name.split(",")[0])
def test_tile_edges(w, precision):
    precision = PRECISIONS[precision]
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    sizes = [1, 127, 129, sms * 128, 4 * sms * 128, 4 * sms * 128 + 1]
    params = synth.random_params(w, 41)
    m = make_model(w, params, sizes[-1], precision=precision)
    for n in sizes:
        pos, u = synth.positions(n, n), synth.sample_uniforms(n, n)
        aux = synth.aux_inputs(n, n) if w.mode == synth.PRODUCT else None
        d, p, _ = m.query_sample(cuda(pos), cuda(u), None if aux is None else cuda(aux))
        m.check_device_status()
        # Every query of the small batches; first, last and a seeded subset of
        # the large ones.
        pick = np.unique(np.r_[0, n - 1, np.random.default_rng(n).choice(n, min(n, 4096), replace=False)])
        gd, gp = host(d)[:, pick].astype(np.float64), host(p)[pick]
        ref = oracle.eval_pdf64(w, params, pos[:, pick], gd, None if aux is None else aux[:, pick])
        if precision in (synth.FP32, synth.FP32_TC):
            assert (np.abs(gp - ref) / ref).max() <= 1e-4, n
        else:
            assert np.quantile(np.abs(gp - ref) / np.maximum(ref, 1e-2 / (4 * math.pi)), 0.999) <= 2e-2, n


def test_fp32_range():
    # Hidden values around 1e20 and weights around 1e-20: FP32 keeps its
    # accuracy over the exponents that a 16-bit format of narrower range
    # would lose.
    w, n = ODD_TWO, 2000
    params = synth.random_params(w, 42)
    ng = sum(synth.grid_sizes(w)) * w.feat
    k = w.widths[0] * w.widths[1]
    params[ng:ng + k] *= np.float32(2.0 ** 66)
    params[ng + k:] *= np.float32(2.0 ** -66)
    pos, u = synth.positions(5, n), synth.sample_uniforms(5, n)
    m = make_model(w, params, n, precision=synth.FP32)
    d, p, _ = m.query_sample(cuda(pos), cuda(u))
    m.check_device_status()
    ref = oracle.eval_pdf64(w, params, pos, host(d).astype(np.float64))
    assert (np.abs(host(p) - ref) / ref).max() <= 1e-4
