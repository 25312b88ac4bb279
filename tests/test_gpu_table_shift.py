"""Grids of two features whose first hashed level starts 1, 2 or 3 entries past
a multiple of four: the library shifts such tables (and gradient, moments and
average with them) so that the hashed levels are aligned. Parameters round
trip, gradients match the oracle (relative L2 1e-4 in FP32, 2e-2 on split
BF16), and one Adam step with the weight average on updates every entry, the
first and the last among them, as the oracle's Adam does from the same
gradient (1e-6, FP32 rounding of one step)."""
import numpy as np
import pytest

import oracle
import synth
from gpu_helpers import cuda, make_model

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _net(first):
    return synth.Workload(name=f"dense {first}, then two hashed levels", mode=synth.RADIANCE,
                          level_res=[first, 30, 45], feat=2, log2_table=12, widths=[8, 16, 8], K=2, lr=1e-2)


# 5^3 = 125: 1 past; 3^3 = 27: 3 past; 6^3 = 216: aligned;
# 125 + 9^3 = 854: 2 past.
NETS = [_net(5), _net(3), _net(6),
        synth.Workload(name="dense 5 and 9, then hashed", mode=synth.RADIANCE, level_res=[5, 9, 30], feat=2,
                       log2_table=12, widths=[8, 16, 8], K=2, lr=1e-2)]


@pytest.mark.parametrize("precision,bar", [(synth.FP32, 1e-4), (synth.BF16X3, 2e-2)], ids=["fp32", "bf16x3"])
@pytest.mark.parametrize("w", NETS, ids=lambda w: w.name.replace(" ", "-"))
def test_shifted_tables(w, precision, bar):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    n = 3000
    params = synth.random_params(w, 61)
    m = make_model(w, params, n, precision=precision)
    assert np.array_equal(m.get_params(), params)
    b = synth.train_batch_uniform(w, n, seed=61)
    dlogv = -(b.radiance.astype(np.float64) / b.pdf) / n
    m.backward(cuda(b.pos), cuda(b.dir), cuda(dlogv))
    g = m.get_grads().astype(np.float64)
    assert np.array_equal(m.grads_device().cpu().numpy().astype(np.float64), g)
    _, ref = oracle.train_grad(w, params, b.pos, b.dir, b.radiance, b.pdf)
    ng = sum(synth.grid_sizes(w)) * w.feat
    for sl in (slice(0, ng), slice(ng, None)):
        assert np.linalg.norm(g[sl] - ref[sl]) <= bar * np.linalg.norm(ref[sl])
    m.set_ema(0.25)
    m.adam_step()
    p, mm, vv = params.astype(np.float64), np.zeros_like(g), np.zeros_like(g)
    oracle.adam(p, g, mm, vv, 1, w.lr, w.beta1, w.beta2, w.eps)
    got = m.get_params()
    # (entries with no gradient stay; a first step moves the others by lr)
    assert np.abs(got - p).max() <= 1e-6
    assert np.abs(m.get_ema_params() - (0.25 * params + 0.75 * got)).max() <= 1e-6
    assert not m.get_grads().any()
    m.check_device_status()


@pytest.mark.parametrize("w", NETS, ids=lambda w: w.name.replace(" ", "-"))
def test_pointers_are_aligned_as_documented(w):
    # 8 bytes, the first hashed level on 32, parameters and gradient alike;
    # the grid and the weights lie where the header says.
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    params = synth.random_params(w, 62)
    m = make_model(w, params, 256)
    sizes = synth.grid_sizes(w)
    dense = sum(s for s, d in zip(sizes, w.level_res) if d ** 3 <= 1 << w.log2_table)
    at, grad = m._L.npm_params_device(m.handle), m._L.npm_grads_device(m.handle)
    assert at % 8 == 0 and (at + 8 * dense) % 32 == 0 and at % 32 == grad % 32
    ng = 2 * sum(sizes)
    mlp = (ng + 63) // 64 * 64

    class Own:
        __cuda_array_interface__ = {"shape": (mlp + params.size - ng,), "typestr": "<f4", "data": (at, False),
                                    "version": 2}

    own = torch.as_tensor(Own(), device="cuda").cpu().numpy()
    assert np.array_equal(own[:ng], params[:ng]) and np.array_equal(own[mlp:], params[ng:])
    m.close()
