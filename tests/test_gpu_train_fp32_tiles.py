"""FP32 training at the edges of its tiles: one sample, a tile less and more
one, more tiles than two groups on every SM hold, on layer widths that fill
the 16-, 32-, 64- and 128-wide register tiles unevenly and lobe counts that
four threads share unevenly. Gradient per tensor (relative L2 1e-4) and loss
(1e-5, FP32 terms summed in 64 bits) against the FP64 oracle."""
import numpy as np
import pytest

import oracle
import synth
from gpu_helpers import cuda, host, make_model

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

NETS = [synth.Workload(name="8-20-68-12", mode=synth.RADIANCE, level_res=[5, 9], feat=4, log2_table=12,
                       widths=[8, 20, 68, 12], K=3),
        synth.Workload(name="28-36-8-product", mode=synth.PRODUCT, level_res=[4, 6, 11], feat=2, log2_table=10,
                       widths=[28, 36, 8], K=2),
        synth.Workload(name="4-100-20", mode=synth.RADIANCE, level_res=[7], feat=3, log2_table=12,
                       widths=[4, 100, 20], K=5)]


@pytest.mark.parametrize("w", NETS, ids=lambda w: w.name)
def test_gradient_and_loss(w):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    sizes = [1, 63, 65, 2 * sms * 64 + 1]
    params = synth.random_params(w, 71)
    m = make_model(w, params, sizes[-1], precision=synth.FP32)
    ng = sum(synth.grid_sizes(w)) * w.feat
    for n in sizes:
        b = synth.train_batch_uniform(w, n, seed=n)
        aux = None if b.aux is None else cuda(b.aux)
        dlogv = -(b.radiance.astype(np.float64) / b.pdf) / n
        m.backward(cuda(b.pos), cuda(b.dir), cuda(dlogv), aux)
        g = m.get_grads().astype(np.float64)
        ref_loss, ref = oracle.train_grad(w, params, b.pos, b.dir, b.radiance, b.pdf, b.aux)
        o = ng
        blocks = [slice(0, ng)]
        for a, c in zip(w.widths[:-1], w.widths[1:]):
            blocks.append(slice(o, o + a * c))
            o += a * c
        for sl in blocks:
            assert np.linalg.norm(g[sl] - ref[sl]) <= 1e-4 * np.linalg.norm(ref[sl]), (n, sl)
        m.set_params(params)
        loss = m.train_step(cuda(b.pos), cuda(b.dir), cuda(b.radiance), cuda(b.pdf), aux)
        assert abs(float(host(loss)[0]) - ref_loss) <= 1e-5 * abs(ref_loss), n
        m.set_params(params)
        m.check_device_status()
