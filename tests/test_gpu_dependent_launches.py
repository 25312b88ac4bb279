"""Training steps and queries back to back, where each kernel may be scheduled
before its predecessor in the stream has finished: densities right after the
last step are those of the parameters it left (FP64 oracle on the parameters
read back; 1e-4 in FP32, else 2e-2 at the 99.9th percentile, denominator
floored at 1e-2 / (4 pi)), and the optimiser has taken every step once (the
loss of each step equals that of a model synchronised after every launch, to
1e-3: the order of the gradient's additions differs). One sample, where most
SMs are idle and the optimiser's blocks wait beside the training kernel, and
many tiles per SM."""
import math

import numpy as np
import pytest

import oracle
import synth
from gpu_helpers import cuda, host, make_model

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

NETS = {"tiny": synth.TINY, "product": synth.PRODUCT_BF16, "own": synth.PAPER_OWN}


@pytest.mark.parametrize("n", [1, 60000])
@pytest.mark.parametrize("net,precision", [("tiny", synth.BF16X3), ("product", synth.BF16X3), ("own", synth.FP32)])
def test_steps_back_to_back(net, precision, n):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    w = NETS[net].with_(precision=precision)
    params = synth.random_params(w, 61)
    b = synth.train_batch_uniform(w, n, seed=61)
    tb = [cuda(v) for v in (b.pos, b.dir, b.radiance, b.pdf)] + [None if b.aux is None else cuda(b.aux)]
    nq = 2000
    pos, u = synth.positions(62, nq), synth.sample_uniforms(62, nq)
    aux = synth.aux_inputs(62, nq) if w.mode == synth.PRODUCT else None
    qa = None if aux is None else cuda(aux)
    qp, qu = cuda(pos), cuda(u)
    m, ref = (make_model(w, params, max(n, nq)) for _ in range(2))
    losses = [m.train_step(*tb) for _ in range(8)]
    d, p, _ = m.query_sample(qp, qu, qa)
    m.check_device_status()
    for loss in losses:
        want = ref.train_step(*tb)
        torch.cuda.synchronize()
        assert abs(float(loss) - float(want)) <= 1e-3 * max(1.0, abs(float(want)))
    want = oracle.eval_pdf64(w, m.get_params(), pos, host(d).astype(np.float64), aux)
    err = np.abs(host(p) - want)
    if precision == synth.FP32:
        assert (err / want).max() <= 1e-4
    else:
        assert np.quantile(err / np.maximum(want, 1e-2 / (4 * math.pi)), 0.999) <= 2e-2
