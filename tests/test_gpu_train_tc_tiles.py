"""Tensor-core training at the edges of its tiles and groups: one sample, a tile
less and more one, one tile for each of two groups on every SM and one more,
on networks whose layers fill the operand planes unevenly, whose gradient and
residuals share an MMA (up to 64 outputs) or not (80), with fewer layers than
levels a thread's deferred scatter has to place, and with one group a CTA.
Gradient per tensor against the FP64 oracle, relative L2 2e-2 (the
reduced-precision bar)."""
import numpy as np
import pytest

import oracle
import synth
from gpu_helpers import cuda, host, make_model

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

NETS = [synth.Workload(name="product-32-20-44-12", mode=synth.PRODUCT, level_res=[4, 6, 9, 14, 20], feat=2,
                       log2_table=12, widths=[32, 20, 44, 12], K=3),
        synth.Workload(name="two-layers-32-64-32", mode=synth.RADIANCE, level_res=[3 + i for i in range(16)], feat=2,
                       log2_table=12, widths=[32, 64, 32], K=8),
        synth.Workload(name="8-80-64-24", mode=synth.RADIANCE, level_res=[6, 30], feat=4, log2_table=13,
                       widths=[8, 80, 64, 24], K=6),
        synth.Workload(name="one-layer-8-8", mode=synth.RADIANCE, level_res=[5, 9, 12], feat=1, log2_table=12,
                       widths=[8, 8], K=2)]


@pytest.mark.parametrize("w", NETS, ids=lambda w: w.name)
def test_gradient(w):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    sizes = [1, 127, 129, 2 * sms * 128, 2 * sms * 128 + 1]
    params = synth.random_params(w, 81)
    m = make_model(w, params, sizes[-1], precision=synth.BF16X3)
    ng = sum(synth.grid_sizes(w)) * w.feat
    for n in sizes:
        b = synth.train_batch_uniform(w, n, seed=n)
        dlogv = -(b.radiance.astype(np.float64) / b.pdf) / n
        m.backward(cuda(b.pos), cuda(b.dir), cuda(dlogv), None if b.aux is None else cuda(b.aux))
        m.check_device_status()
        g = m.get_grads().astype(np.float64)
        ref_loss, ref = oracle.train_grad(w, params, b.pos, b.dir, b.radiance, b.pdf, b.aux)
        o, blocks = ng, [slice(0, ng)]
        for a, c in zip(w.widths[:-1], w.widths[1:]):
            blocks.append(slice(o, o + a * c))
            o += a * c
        for sl in blocks:
            assert np.linalg.norm(g[sl] - ref[sl]) <= 2e-2 * np.linalg.norm(ref[sl]), (n, sl)
        loss = m.train_step(cuda(b.pos), cuda(b.dir), cuda(b.radiance), cuda(b.pdf),
                            None if b.aux is None else cuda(b.aux))
        assert abs(float(host(loss)[0]) - ref_loss) <= 2e-2 * abs(ref_loss) + 1e-3, n
        m.set_params(params)
