"""Corner blocks of the dense levels (read by batches of 2^18 queries and
more): the same bytes as the table, so a large batch gives exactly what the
table gives its two halves, on every table format, with levels of the
smallest resolutions and hashed levels between; and they follow the
parameters through set_params, a training step, the weight average, a write
through npm_params_device (in graphs captured before the address was asked for
too) and a query on another stream beside an update; memory only for handles
and servers whose batches are large enough."""
import numpy as np
import pytest

import synth
from gpu_helpers import cuda, make_model

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

N = 1 << 18
TWO = synth.Workload(name="6 levels x 2 feats", mode=synth.RADIANCE, level_res=[2, 3, 40, 10, 17, 25], feat=2,
                     log2_table=14, widths=[12, 32, 16], K=4, n_train=4096)
FOUR = synth.Workload(name="4 levels x 4 feats", mode=synth.RADIANCE, level_res=[30, 2, 9, 20], feat=4,
                      log2_table=13, widths=[16, 32, 16], K=4, n_train=4096)


def _same(m, pos, u):
    d, p, _ = m.query_sample(pos, u, n=N)
    for a, b in ((0, N // 2), (N // 2, N)):
        dh, ph, _ = m.query_sample(pos[:, a:b].contiguous(), u[:, a:b].contiguous())
        assert torch.equal(d[:, a:b], dh) and torch.equal(p[a:b], ph), (a, b)


@pytest.mark.parametrize("precision", [synth.FP32, synth.FP32_TC, synth.BF16X3, synth.FP16],
                         ids=["fp32", "fp32tc", "bf16x3", "fp16"])
@pytest.mark.parametrize("w", [TWO, FOUR], ids=lambda w: w.name)
def test_blocks_equal_the_table(w, precision):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    x = synth.positions(3, N)
    x[:, :8] = np.array([[0, 1, 0.5, 1, 0, 0.9999999, 1e-7, 0.25]] * 3, dtype=np.float32)  # edges of the box
    pos, u = cuda(x), cuda(synth.sample_uniforms(3, N))
    m = make_model(w, synth.random_params(w, 51), N, precision=precision)
    _same(m, pos, u)
    m.set_params(synth.random_params(w, 52))
    _same(m, pos, u)
    b = synth.train_batch_uniform(w, w.n_train, seed=51)
    m.train_step(cuda(b.pos), cuda(b.dir), cuda(b.radiance), cuda(b.pdf))
    _same(m, pos, u)
    m.set_ema(0.5)
    m.train_step(cuda(b.pos), cuda(b.dir), cuda(b.radiance), cuda(b.pdf))
    _same(m, pos, u)
    m.set_ema(0.0)
    # The FP32 tables are the parameters: a write through their address counts.
    ptr = m._L.npm_params_device(m.handle)
    ng = sum(synth.grid_sizes(w)) * w.feat

    class Grid:
        __cuda_array_interface__ = {"shape": (ng,), "typestr": "<f4", "data": (ptr, False), "version": 2}

    torch.as_tensor(Grid(), device="cuda").mul_(0.5)
    _same(m, pos, u)
    m.check_device_status()
    m.close()


@pytest.mark.parametrize("precision", [synth.FP32, synth.FP32_TC], ids=["fp32", "fp32tc"])
def test_write_through_the_address_reaches_an_earlier_capture(precision):
    # A query captured before the parameters' address was first asked for
    # reads, at each replay, what has been written through it.
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    w = TWO
    pos, u = cuda(synth.positions(5, N)), cuda(synth.sample_uniforms(5, N))
    m = make_model(w, synth.random_params(w, 53), N, precision=precision)
    out = torch.empty(3, N, device="cuda"), torch.empty(N, device="cuda")
    m.query_sample(pos, u, out=out)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        m.query_sample(pos, u, out=out)
    ptr = m._L.npm_params_device(m.handle)
    ng = sum(synth.grid_sizes(w)) * w.feat

    class Grid:
        __cuda_array_interface__ = {"shape": (ng,), "typestr": "<f4", "data": (ptr, False), "version": 2}

    grid = torch.as_tensor(Grid(), device="cuda")
    for scale in (0.5, -1.0):
        grid.mul_(scale)
        graph.replay()
        for a, b in ((0, N // 2), (N // 2, N)):
            d, p, _ = m.query_sample(pos[:, a:b].contiguous(), u[:, a:b].contiguous())
            assert torch.equal(out[0][:, a:b], d) and torch.equal(out[1][a:b], p), (scale, a)
    m.check_device_status()
    m.close()


def test_address_asked_for_during_a_capture():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    w = TWO
    pos, u = cuda(synth.positions(6, 4096)), cuda(synth.sample_uniforms(6, 4096))
    m = make_model(w, synth.random_params(w, 54), 4096, precision=synth.FP32)
    out = torch.empty(3, 4096, device="cuda"), torch.empty(4096, device="cuda")
    want = m.query_sample(pos, u)[1]
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        m.query_sample(pos, u, out=out)
        assert m._L.npm_params_device(m.handle)
    graph.replay()
    assert torch.equal(out[1], want)
    m.close()


def test_query_beside_an_update_leaves_no_stale_blocks():
    # A query on another stream while the parameters are being replaced may
    # see either set; the next query ordered after both sees the new one. The
    # second stream's delay walks over the update's launches.
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    w = synth.Workload(name="dense 40, then 12 levels of 2^20", mode=synth.RADIANCE, level_res=[40] + [128] * 12,
                       feat=2, log2_table=20, widths=[28, 16, 8], K=2, n_train=4096)
    pos, u = cuda(synth.positions(7, N)), cuda(synth.sample_uniforms(7, N))
    sets = [cuda(synth.random_params(w, s)) for s in (55, 56)]
    m = make_model(w, synth.random_params(w, 57), N, precision=synth.FP16)
    _same(m, pos, u)
    side = torch.cuda.Stream()
    out = torch.empty(3, N, device="cuda"), torch.empty(N, device="cuda")
    for i in range(60):
        torch.cuda.synchronize()
        with torch.cuda.stream(side):
            torch.cuda._sleep(1 + 4000 * i)  # 2 us a step
            m.query_sample(pos, u, out=out)
        m.set_params_device(sets[i & 1])
        torch.cuda.synchronize()
        _same(m, pos, u)
    m.check_device_status()
    m.close()


def _used(make):
    """Device memory that an object takes, in MB (rounded by the driver)."""
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    made = make()
    torch.cuda.synchronize()
    return (before - torch.cuda.mem_get_info()[0]) / 2 ** 20, made


def test_memory_only_where_batches_are_large_enough():
    # 33 MB on this grid: a handle for smaller batches has none, until a
    # server gathers larger ones from them.
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_2504_04315_gb300 as npm
    w = synth.PAPER_HASH
    make = {n: (lambda n=n: npm.NPM(npm.config_from(w, max_batch=n))) for n in (N - 1, N)}
    make[N]().close()  # (the context's and the driver's own memory)
    small, m = _used(make[N - 1])
    large, big = _used(make[N])
    big.close()
    assert 24 < large - small < 48, (small, large)
    first, server = _used(lambda: npm.Server(m, 2 * N))
    server.close()
    second, server = _used(lambda: npm.Server(m, 2 * N))
    server.close()
    assert 24 < first - second < 48, (first, second)
    params = synth.random_params(w, 58)
    m.set_params(params)
    # Four requests of 2^17 queries that the server takes in one launch give
    # what the model gives one of them.
    n = N // 2
    pos, u = synth.positions(8, n), synth.sample_uniforms(8, n)
    want = m.query_sample(cuda(pos), cuda(u))[1].cpu()
    with npm.Server(m, 2 * N) as s:
        t = torch.from_numpy(pos).pin_memory(), torch.from_numpy(u).pin_memory()
        out = [(torch.zeros(3, n).pin_memory(), torch.zeros(n).pin_memory()) for _ in range(4)]
        s.hold(True)
        tickets = [s.submit_query(t[0], t[1], d, p) for d, p in out]
        s.hold(False)
        for k in tickets:
            s.wait(k)
        for _, p in out:
            assert torch.equal(p, want)
    m.close()
