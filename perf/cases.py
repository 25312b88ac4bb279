"""Performance cases of the guiding library: what a renderer has it do, call by call.

A case names one public entry point (`op`), one network of the repository's
workloads (`net`), an arithmetic (`prec`) and a batch size (`n`):

  sample  NPM.query_sample       directions and densities of a wavefront of path vertices
  host    NPM.query_sample_host  the same from and to pinned host buffers
  pdf     NPM.eval_pdf           densities at given directions (multiple importance sampling)
  logpdf  NPM.eval_log_pdf       the same as logarithms
  train   NPM.train_step         one step of online training: loss, gradient, Adam
  grad    log_density            autograd: log densities and the parameters' gradient

`run` makes one pass through the entry point; `exact` states in 64-bit torch
what it computes, written from the method: grid blend, SH inputs, MLP, lobe
mapping, vMF sampling and density, weighted log-likelihood, Adam.
"""
from __future__ import annotations

import math

import torch

import paper_2504_04315_gb300 as npm

RES16 = [16, 20, 25, 32, 40, 50, 64, 80, 101, 128, 161, 203, 256, 322, 406, 512]
RES8 = [8, 11, 15, 22, 31, 43, 61, 86]

# The networks of the repository's workloads.
NETS = {
    # the serving network: one dense level, three narrow layers, four lobes
    "tiny": dict(mode=npm.RADIANCE, res=[16], feat=4, log2=19, widths=[4, 32, 32, 16], K=4, lr=5e-3),
    # 16-level hash grid, four 64-wide layers, eight lobes
    "paper_hash": dict(mode=npm.RADIANCE, res=RES16, feat=2, log2=19, widths=[32, 64, 64, 64, 32], K=8, lr=5e-3),
    # the paper's own shape: eight dense levels of four features
    "paper_own": dict(mode=npm.RADIANCE, res=RES8, feat=4, log2=20, widths=[32, 64, 64, 64, 32], K=8, lr=5e-3),
    # product mode: the hash grid plus outgoing direction, normal and roughness
    "product": dict(mode=npm.PRODUCT, res=RES16, feat=2, log2=19, widths=[64, 64, 64, 64, 32], K=8, lr=1e-2),
}
PREC = {"fp32": npm.FP32, "fp32tc": npm.FP32_TC, "bf16x3": npm.BF16X3, "fp16": npm.FP16}
BETA1, BETA2, EPS = 0.9, 0.99, 1e-8
ADAM_STEP = 300  # completed steps of the training run that a train case continues


def listed():
    return [
        # The repository's headline: a wavefront of 2^20 vertices on the
        # paper-shaped hash grid in FP32, the default arithmetic.
        dict(name="sample_paper_hash_fp32", op="sample", net="paper_hash", prec="fp32", n=1 << 20, pad=0, ufrac=0.0),
        # The FP32-accuracy tensor-core mode, product sampling, a compacted
        # queue (an odd length inside a longer buffer).
        dict(name="sample_product_fp32tc", op="sample", net="product", prec="fp32tc", n=300007, pad=1701, ufrac=0.0),
        # A whole 1080p frame's first bounce with the 50 % BSDF stand-in, FP16.
        dict(name="sample_paper_hash_fp16", op="sample", net="paper_hash", prec="fp16", n=1920 * 1080, pad=0, ufrac=0.5),
        # The serving network's large reduced-precision batch.
        dict(name="sample_tiny_bf16x3", op="sample", net="tiny", prec="bf16x3", n=1 << 22, pad=0, ufrac=0.0),
        # The last bounces of a frame: a few live paths, where the launch counts.
        dict(name="sample_tiny_fp16_small", op="sample", net="tiny", prec="fp16", n=1000, pad=24, ufrac=0.5),
        # A renderer whose queues live on the host.
        dict(name="host_paper_hash_bf16x3", op="host", net="paper_hash", prec="bf16x3", n=1 << 20, pad=0, ufrac=0.0),
        # MIS weights of BSDF samples: densities at given directions, on the
        # paper's own network shape.
        dict(name="pdf_paper_own_bf16x3", op="pdf", net="paper_own", prec="bf16x3", n=250007, pad=0, ufrac=0.0),
        # A small tile's log densities in FP32 (a preview or probe update).
        dict(name="logpdf_paper_hash_fp32_small", op="logpdf", net="paper_hash", prec="fp32", n=3001, pad=0, ufrac=0.0),
        # The training workload: product mode, 2^19 samples, Adam over the
        # 10 M parameters.
        dict(name="train_product_bf16x3", op="train", net="product", prec="bf16x3", n=1 << 19, pad=0, ufrac=0.0),
        # The serving frame's training batch.
        dict(name="train_tiny_bf16x3", op="train", net="tiny", prec="bf16x3", n=1 << 18, pad=0, ufrac=0.0),
        # Training in the default arithmetic on the paper's own network shape.
        dict(name="train_paper_own_fp32", op="train", net="paper_own", prec="fp32", n=65551, pad=0, ufrac=0.0),
        # The differentiable wrapper inside a torch program, FP32.
        dict(name="grad_product_fp32", op="grad", net="product", prec="fp32", n=20011, pad=0, ufrac=0.0),
    ]


def draw(rng):
    """One more case: any entry point, network and arithmetic, sizes spread over
    their logarithm from a few hundred to the largest listed for that use."""
    op = rng.choice(["sample", "sample", "sample", "host", "pdf", "logpdf", "train", "train", "grad"])
    net = rng.choice(list(NETS))
    prec = rng.choice(list(PREC))
    if op in ("sample", "host", "pdf", "logpdf"):
        top = {"tiny": 22.0, "paper_hash": 20.9, "paper_own": 20.9, "product": 20.0}[net]
    elif op == "train":
        top = {"tiny": 20.0, "paper_hash": 18.9, "paper_own": 18.9, "product": 18.9}[net]
    else:
        top = 17.0
    n = max(257, int(2.0 ** rng.uniform(8.0, top)))
    return dict(op=op, net=net, prec=prec, n=n, pad=rng.choice([0, 0, 1, 37, 1000]),
                ufrac=rng.choice([0.0, 0.5]) if op in ("sample", "host") else 0.0)


# ------------------------------------------------------------------ inputs


def _generator(seed, stream):
    return torch.Generator(device="cuda").manual_seed((int(seed) * 1000003 + stream) & 0x7FFFFFFFFFFFFFFF)


def _uniform(g, *shape):
    return torch.rand(*shape, generator=g, device="cuda", dtype=torch.float32)


def _sphere(u):
    """Uniform unit vectors [3][n] (64-bit) from uniforms [2][n]."""
    u = u.double()
    z = 1.0 - 2.0 * u[0]
    r = torch.sqrt(torch.clamp(1.0 - z * z, min=0.0))
    return torch.stack([r * torch.cos(2 * math.pi * u[1]), r * torch.sin(2 * math.pi * u[1]), z])


def _grid_sizes(net):
    return [min(1 << net["log2"], d ** 3) for d in net["res"]]


def _inputs_width(net):
    return len(net["res"]) * net["feat"] + (21 if net["mode"] == npm.PRODUCT else 0)


def _params(net, seed):
    """Parameters that decode like a trained model (uneven weights, lobes all
    over the sphere, kappa up to tens), public layout."""
    g = _generator(seed, 1)
    parts = [_uniform(g, sum(_grid_sizes(net)) * net["feat"]) * 2.0 - 1.0]
    w, ew = net["widths"], _inputs_width(net)
    for i in range(len(w) - 1):
        a = 2.0 * math.sqrt(6.0 / ((min(w[0], ew) if i == 0 else w[i]) + w[i + 1]))
        m = (_uniform(g, w[i + 1], w[i]) * 2.0 - 1.0) * a
        if i == 0:
            m[:, ew:] = 0.0  # the padding of the inputs
        if i == len(w) - 2:
            m[1::4] *= 6.0  # the rows of kappa
        parts.append(m.reshape(-1))
    return torch.cat(parts)


def _aux(g, n):
    """Product-mode inputs [7][n]: outgoing direction on the normal's
    hemisphere, normal, roughness."""
    u = _uniform(g, 5, n)
    nrm, wo = _sphere(u[0:2]), _sphere(u[2:4])
    wo = torch.where((nrm * wo).sum(0) < 0, -wo, wo)
    return torch.cat([wo, nrm, (0.05 + 0.95 * u[4].double())[None]]).float()


def _radiance(x, w, aux):
    """The stand-in scene's radiance: three lobes whose means and sharpness
    vary with position, times a glossy factor in product mode (64-bit)."""
    x, w = x.double(), w.double()
    axes = [(0.0, 0.0, 1.0), (1.0, 0.0, 0.0), tuple(v / math.sqrt(3.0) for v in (-1.0, -1.0, 1.0))]
    out = torch.zeros_like(x[0])
    for m, (amp, e) in enumerate(zip((0.5, 0.3, 0.2), axes)):
        mu = torch.stack([e[0] + 0.5 * torch.sin(2 * math.pi * x[1] + m),
                          e[1] + 0.5 * torch.sin(2 * math.pi * x[2] + 2 * m),
                          e[2] + 0.5 * torch.sin(2 * math.pi * x[0] + 3 * m)])
        mu = mu / mu.norm(dim=0)
        k = 1.0 + 49.0 * (0.5 + 0.5 * torch.sin(2 * math.pi * (m + 1) * x.sum(0) / 3.0 + m))
        out += amp * k / (2 * math.pi * -torch.expm1(-2 * k)) * torch.exp(k * ((mu * w).sum(0) - 1.0))
    if aux is not None:
        wo, nrm, a2 = aux[0:3].double(), aux[3:6].double(), aux[6].double() ** 4
        h = w + wo
        ch = (nrm * h).sum(0) / h.norm(dim=0).clamp(min=1e-9)
        gloss = torch.where(ch > 0, a2 * a2 / (ch * ch * (a2 - 1.0) + 1.0) ** 2, torch.zeros_like(ch))
        out *= (nrm * w).sum(0).clamp(min=0.0) * (0.3 + 0.7 * gloss)
    return out


def _padded(t, pad):
    """[rows][n] -> [rows][n + pad]: the live part of a longer buffer."""
    return torch.nn.functional.pad(t, (0, pad)).contiguous() if pad else t.contiguous()


# Queries whose sample is a matter of rounding are not drawn: u0 this close to
# a cumulative weight (two neighbouring lobes), or the chosen lobe's mean this
# close to the equator (the two branches of the sampling frame, whose azimuths
# differ). Any two correct implementations differ there by a whole direction.
_MARGIN = {"fp32": 1e-4, "fp32tc": 1e-4, "bf16x3": 1e-3, "fp16": 4e-3}


def _query_inputs(case, seed, params):
    """pos, aux, u on the device for a sampling case."""
    net, n = NETS[case["net"]], case["n"]
    rows = 4 if case["ufrac"] > 0 else 3
    g = _generator(seed, 2)
    kept, have = [], 0
    while have < n:
        m = n - have + (n - have) // 8 + 64
        pos, u = _uniform(g, 3, m), _uniform(g, rows, m)
        aux = _aux(g, m) if net["mode"] == npm.PRODUCT else None
        ok = torch.empty(m, dtype=torch.bool, device="cuda")
        for a in range(0, m, 1 << 18):
            b = slice(a, min(m, a + (1 << 18)))
            lam, _, mu, _ = _mixture(net, params, pos[:, b], None if aux is None else aux[:, b], torch.float32)
            cum = torch.cumsum(lam, 1)
            mg = _MARGIN[case["prec"]]
            far = ((cum[:, :-1] - u[0, b][:, None]).abs() > mg).all(1) & (u[0, b] < 1.0 - mg)
            z = mu[torch.arange(mu.shape[0], device="cuda"), _lobe_of(cum, u[0, b])][:, 2]
            ok[b] = far & (z.abs() > mg)
        kept.append((pos[:, ok], None if aux is None else aux[:, ok], u[:, ok]))
        have += int(ok.sum())
    cat = [None if kept[0][i] is None else torch.cat([k[i] for k in kept], 1)[:, :n].contiguous() for i in range(3)]
    return cat[0], cat[1], cat[2]


def _eval_inputs(case, seed):
    net, n = NETS[case["net"]], case["n"]
    g = _generator(seed, 3)
    aux = _aux(g, n) if net["mode"] == npm.PRODUCT else None
    return _uniform(g, 3, n), aux, _sphere(_uniform(g, 2, n)).float()


def _train_inputs(case, seed):
    """Uniform directions, the scene's radiance times Exponential(1) noise."""
    net = NETS[case["net"]]
    pos, aux, d = _eval_inputs(case, seed)
    noise = -torch.log1p(-_uniform(_generator(seed, 4), case["n"]).double())
    rad = (_radiance(pos, d, aux) * noise).float()
    return pos, aux, d, rad, torch.full_like(rad, 1.0 / (4.0 * math.pi))


def _adam_state(net, seed):
    """Moments of a run in progress: the second one around the square of the
    gradients that such batches give (1e-6 per grid entry, 1e-2 per weight),
    spread over a decade; the first one within it."""
    g = _generator(seed, 5)
    ng = sum(_grid_sizes(net)) * net["feat"]
    np_ = ng + sum(a * b for a, b in zip(net["widths"][:-1], net["widths"][1:]))
    s = torch.pow(10.0, _uniform(g, np_) - 0.5)
    s[:ng] *= 1e-6
    s[ng:] *= 1e-2
    return (_uniform(g, np_) - 0.5) * s, s * s


class _Shared:
    """A library-owned FP32 device buffer as a torch tensor. The tensor keeps
    this object, and with it the model that owns the buffer, alive."""

    def __init__(self, model, ptr, count):
        self.model = model
        self.__cuda_array_interface__ = {"shape": (count,), "typestr": "<f4", "data": (ptr, False), "version": 2}


def _model(case, params):
    net = NETS[case["net"]]
    m = npm.NPM(npm.make_config(net["mode"], net["res"], net["feat"], net["log2"], net["widths"], net["K"],
                                precision=PREC[case["prec"]], lr=net["lr"], beta1=BETA1, beta2=BETA2, eps=EPS,
                                max_batch=case["n"] + case["pad"]))
    m.set_params_device(params)
    return m


def prepare(case, seed):
    net, n, pad = NETS[case["net"]], case["n"], case["pad"]
    params = _params(net, seed)
    s = {"case": case, "model": _model(case, params)}
    if case["op"] in ("sample", "host"):
        pos, aux, u = (None if t is None else _padded(t, pad) for t in _query_inputs(case, seed, params))
        out = (torch.zeros(3, n + pad, device="cuda"), torch.zeros(n + pad, device="cuda"))
        if case["op"] == "host":
            pos, aux, u = (None if t is None else t.cpu().pin_memory() for t in (pos, aux, u))
            out = tuple(t.cpu().pin_memory() for t in out)
        s.update(pos=pos, aux=aux, u=u, out=out)
    elif case["op"] in ("pdf", "logpdf"):
        s["pos"], s["aux"], s["dir"] = (None if t is None else _padded(t, pad) for t in _eval_inputs(case, seed))
    elif case["op"] == "train":
        pos, aux, d, rad, pdf = _train_inputs(case, seed)
        s["pos"], s["aux"], s["dir"] = (None if t is None else _padded(t, pad) for t in (pos, aux, d))
        s["rad"], s["pdf"] = rad, pdf
        m, v = _adam_state(net, seed)
        s["model"].set_adam(ADAM_STEP, m.cpu().numpy(), v.cpu().numpy())
        # The library's parameters, where the step leaves the updated ones:
        # the grid, then the MLP from the next multiple of 64 values.
        ng = sum(_grid_sizes(net)) * net["feat"]
        at = (ng + 63) // 64 * 64
        lib, model = s["model"]._L, s["model"]
        own = torch.as_tensor(_Shared(model, lib.npm_params_device(model.handle), at + params.numel() - ng), device="cuda")
        s["grid"], s["mlp"] = own[:ng], own[at:]
    else:
        s["pos"], s["aux"], s["dir"], rad, pdf = _train_inputs(case, seed)
        s["theta"] = params.requires_grad_(True)
        s["weight"] = -rad / (pdf * n)
    torch.cuda.synchronize()
    return s


def run(s):
    case, m = s["case"], s["model"]
    n, op = case["n"], case["op"]
    if op == "sample":
        d, p, _ = m.query_sample(s["pos"], s["u"], s["aux"], uniform_frac=case["ufrac"], n=n, out=s["out"])
        return {"dir": d[:, :n], "pdf": p[:n]}
    if op == "host":
        d, p = s["out"]
        m.query_sample_host(s["pos"], s["u"], d, p, aux=s["aux"], uniform_frac=case["ufrac"], n=n)
        return {"dir": d[:, :n], "pdf": p[:n]}
    if op == "pdf":
        return m.eval_pdf(s["pos"], s["dir"], s["aux"], n=n)[:n]
    if op == "logpdf":
        return m.eval_log_pdf(s["pos"], s["dir"], s["aux"], n=n)[:n]
    if op == "train":
        loss = m.train_step(s["pos"], s["dir"], s["rad"], s["pdf"], s["aux"], n=n)
        return {"loss": loss, "grid": s["grid"], "mlp": s["mlp"]}
    lv = npm.log_density(s["theta"], m, s["pos"], s["dir"], s["aux"])
    (g,) = torch.autograd.grad(lv, s["theta"], s["weight"])
    return {"logv": lv, "grad": g}


# ------------------------------------------------------- the method in torch


def _encode(net, grid, pos):
    """Trilinear blend of every level's eight corner features, [n][L F]."""
    feats, off = [], 0
    x = torch.clamp(pos.float(), 0.0, 1.0)
    T = 1 << net["log2"]
    for D, size in zip(net["res"], _grid_sizes(net)):
        level = grid[off * net["feat"]:(off + size) * net["feat"]].reshape(size, net["feat"])
        off += size
        p = x * float(D - 1)  # the lattice coordinate is one FP32 multiply
        cell = torch.clamp(torch.floor(p).long(), max=D - 2)
        f = (p - cell.float()).to(grid.dtype)
        acc = 0.0
        for c in range(8):
            b = (c & 1, (c >> 1) & 1, (c >> 2) & 1)
            i, j, k = (cell[a] + b[a] for a in range(3))
            if D ** 3 <= T:
                idx = i + D * (j + D * k)
            else:
                idx = (i ^ (j * 2654435761 & 0xFFFFFFFF) ^ (k * 805459861 & 0xFFFFFFFF)) & (T - 1)
            w = 1.0
            for a in range(3):
                w = w * (f[a] if b[a] else 1.0 - f[a])
            acc = acc + w[:, None] * level[idx]
        feats.append(acc)
    return torch.cat(feats, 1)


def _sh(aux, dt):
    """Real SH of the outgoing direction (4 bands) and normal (2 bands), and
    the roughness, [n][21]."""
    x, y, z = (aux[i].to(dt) for i in range(3))
    nx, ny, nz, r = (aux[3 + i].to(dt) for i in range(4))
    p = math.pi
    c0, c1 = 0.5 * math.sqrt(1 / p), math.sqrt(3 / (4 * p))
    out = [c0 + 0 * x, c1 * y, c1 * z, c1 * x,
           0.5 * math.sqrt(15 / p) * x * y, 0.5 * math.sqrt(15 / p) * y * z, 0.25 * math.sqrt(5 / p) * (3 * z * z - 1),
           0.5 * math.sqrt(15 / p) * x * z, 0.25 * math.sqrt(15 / p) * (x * x - y * y),
           0.25 * math.sqrt(35 / (2 * p)) * y * (3 * x * x - y * y), 0.5 * math.sqrt(105 / p) * x * y * z,
           0.25 * math.sqrt(21 / (2 * p)) * y * (5 * z * z - 1), 0.25 * math.sqrt(7 / p) * z * (5 * z * z - 3),
           0.25 * math.sqrt(21 / (2 * p)) * x * (5 * z * z - 1), 0.25 * math.sqrt(105 / p) * z * (x * x - y * y),
           0.25 * math.sqrt(35 / (2 * p)) * x * (x * x - 3 * y * y),
           c0 + 0 * nx, c1 * ny, c1 * nz, c1 * nx, r]
    return torch.stack(out, 1)


def _mixture(net, params, pos, aux, dt):
    """lam, kap [n][K], mu [n][K][3] and log lam of the decoded mixtures."""
    ng = sum(_grid_sizes(net)) * net["feat"]
    h = _encode(net, params[:ng].to(dt), pos)
    if aux is not None:
        h = torch.cat([h, _sh(aux, dt)], 1)
    w, o = net["widths"], ng
    if h.shape[1] < w[0]:
        h = torch.nn.functional.pad(h, (0, w[0] - h.shape[1]))
    for i in range(len(w) - 1):
        h = h @ params[o:o + w[i] * w[i + 1]].to(dt).reshape(w[i + 1], w[i]).T
        o += w[i] * w[i + 1]
        if i < len(w) - 2:
            h = torch.relu(h)
    raw = h.reshape(-1, net["K"], 4)
    loglam = torch.log_softmax(raw[..., 0], 1)
    kap = torch.nn.functional.softplus(raw[..., 1], threshold=1e9)
    th, ph = math.pi * torch.sigmoid(raw[..., 2]), 2 * math.pi * torch.sigmoid(raw[..., 3])
    mu = torch.stack([torch.sin(th) * torch.cos(ph), torch.sin(th) * torch.sin(ph), torch.cos(th)], -1)
    return loglam.exp(), kap, mu, loglam


def _log_v(mix, d):
    """log of the mixture density at directions d [3][n]."""
    _, kap, mu, loglam = mix
    c = torch.log(kap / (2 * math.pi * -torch.expm1(-2 * kap)))
    return torch.logsumexp(loglam + c + kap * ((mu * d.T.to(mu.dtype)[:, None, :]).sum(-1) - 1.0), 1)


def _lobe_of(cum, u0):
    """Smallest lobe whose cumulative weight exceeds u0."""
    return torch.clamp((u0[:, None] >= cum[:, :-1]).sum(1), max=cum.shape[1] - 1)


def _sample(mix, u, ufrac):
    """Directions [3][n] and strategy densities [n]."""
    lam, kap, mu, _ = mix
    u = u.to(lam.dtype)
    at = torch.arange(lam.shape[0], device=lam.device)
    i = _lobe_of(torch.cumsum(lam, 1), u[0])
    k, m = kap[at, i], mu[at, i]
    t = torch.clamp(-torch.log1p(u[1] * torch.expm1(-2 * k)) / k, 0.0, 2.0)  # 1 - cosine to the mean
    s, phi = torch.sqrt(t * (2.0 - t)), 2 * math.pi * u[2]
    sg = torch.where(m[:, 2] >= 0, 1.0, -1.0).to(lam.dtype)
    a = -1.0 / (sg + m[:, 2])
    b = m[:, 0] * m[:, 1] * a
    tx = torch.stack([1.0 + sg * m[:, 0] ** 2 * a, sg * b, -sg * m[:, 0]])
    ty = torch.stack([b, sg + m[:, 1] ** 2 * a, -m[:, 1]])
    d = s * torch.cos(phi) * tx + s * torch.sin(phi) * ty + (1.0 - t) * m.T
    if ufrac > 0:
        z = 1.0 - 2.0 * u[1]
        r = torch.sqrt(torch.clamp(1.0 - z * z, min=0.0))
        d = torch.where(u[3] < ufrac, torch.stack([r * torch.cos(phi), r * torch.sin(phi), z]), d)
    return d, ufrac / (4 * math.pi) + (1.0 - ufrac) * _log_v(mix, d).exp()


def exact(case, seed):
    net, n, op = NETS[case["net"]], case["n"], case["op"]
    params = _params(net, seed)
    p64 = params.double()
    if op in ("sample", "host"):
        pos, aux, u = _query_inputs(case, seed, params)
    elif op in ("pdf", "logpdf"):
        pos, aux, d = _eval_inputs(case, seed)
    else:
        pos, aux, d, rad, pdf = _train_inputs(case, seed)
        weight = -rad.double() / (pdf.double() * n)
        p64.requires_grad_(True)
    outs, loss = [], 0.0
    for a in range(0, n, 1 << 17):
        b = slice(a, min(n, a + (1 << 17)))
        mix = _mixture(net, p64, pos[:, b], None if aux is None else aux[:, b], torch.float64)
        if op in ("sample", "host"):
            outs.append(_sample(mix, u[:, b], case["ufrac"]))
        else:
            lv = _log_v(mix, d[:, b])
            if op in ("train", "grad"):
                (weight[b] * lv).sum().backward()
                loss = loss + (weight[b] * lv).sum().detach()
            outs.append(lv.detach())
    if op in ("sample", "host"):
        return {"dir": torch.cat([o[0] for o in outs], 1), "pdf": torch.cat([o[1] for o in outs])}
    lv = torch.cat(outs)
    if op == "pdf":
        return lv.exp()
    if op == "logpdf":
        return lv
    if op == "grad":
        return {"logv": lv, "grad": p64.grad}
    m, v = (t.double() for t in _adam_state(net, seed))
    g, t = p64.grad, ADAM_STEP + 1
    m, v = BETA1 * m + (1 - BETA1) * g, BETA2 * v + (1 - BETA2) * g * g
    new = params.double() - net["lr"] * (m / (1 - BETA1 ** t)) / (torch.sqrt(v / (1 - BETA2 ** t)) + EPS)
    ng = sum(_grid_sizes(net)) * net["feat"]
    return {"loss": loss.reshape(1), "grid": new[:ng], "mlp": new[ng:]}


# ------------------------------------------------------ work and tolerance


def work(case):
    net, n, op = NETS[case["net"]], case["n"], case["op"]
    w, L, F = net["widths"], len(net["res"]), net["feat"]
    mlp = sum(a * b for a, b in zip(w[:-1], w[1:]))
    grid = sum(_grid_sizes(net)) * F
    fwd = n * (2 * mlp + 16 * L * F)
    aux = 7 if net["mode"] == npm.PRODUCT else 0
    table = min(grid, 8 * L * F * n) * (2 if case["prec"] in ("bf16x3", "fp16") else 4) + 4 * mlp
    if op in ("sample", "host"):
        return {"bytes": table + 4 * n * (3 + aux + (4 if case["ufrac"] > 0 else 3) + 4), "flops": fwd}
    if op in ("pdf", "logpdf"):
        return {"bytes": table + 4 * n * (3 + aux + 3 + 1), "flops": fwd}
    if op == "train":  # parameters and both moments read and written
        return {"bytes": 24 * (grid + mlp) + 4 * n * (3 + aux + 3 + 2) + 4, "flops": 3 * fwd + 12 * (grid + mlp)}
    # theta read, its gradient written, log densities out and their weights in
    return {"bytes": 8 * (grid + mlp) + 4 * n * (3 + aux + 3 + 2), "flops": 3 * fwd}


# About four times the largest differences from exact() over 160 cases of
# these ranges. FP32 and the FP32-accuracy mode: hardware exponentials at
# arguments up to tens, directions near the frame's branches. Split BF16 and
# FP16: the operands' rounding, amplified by sharp lobes; FP16 tables hold
# the grid. Training: largest where a gradient that cancels to nothing meets
# a small second moment.
_TOLERANCE = {
    "sample": {"fp32": (3e-5, 1e-2), "fp32tc": (6e-5, 8e-2), "bf16x3": (1.7e-3, 4e-2), "fp16": (4e-3, 0.13)},
    "pdf": {"fp32": (2e-5, 1e-4), "fp32tc": (2e-5, 1e-4), "bf16x3": (3e-3, 5e-2), "fp16": (6e-3, 8e-2)},
    "logpdf": {"fp32": (3e-6, 2e-5), "fp32tc": (3e-6, 2e-5), "bf16x3": (8e-4, 1e-2), "fp16": (2.2e-3, 2.8e-2)},
    "train": {"fp32": (1.1e-5, 1e-3), "fp32tc": (1.1e-5, 1e-3), "bf16x3": (3.2e-4, 4.5e-2), "fp16": (3.2e-4, 4.5e-2)},
    "grad": {"fp32": (1.3e-5, 3.3e-3), "fp32tc": (1.3e-5, 3.3e-3), "bf16x3": (7e-3, 0.75), "fp16": (7e-3, 0.75)},
}


def tolerance(case):
    rel, most = _TOLERANCE["sample" if case["op"] == "host" else case["op"]][case["prec"]]
    return {"rel": rel, "max": most}
