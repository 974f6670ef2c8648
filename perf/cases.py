"""What the library is measured on: the calls a localisation program makes, over the range of
sizes it makes them in.

Sizes are those of the workloads of ``bench.py`` and the tests: single filter steps from 32
particles x 8 pixels up to 600 x 64, maps read point by point, whole localisation runs of 1 to 16
queries, and the gradients that fitting a map or a proposal takes.

* ``query``          colour and density of the map at points (one pass of the NeRF MLP)
* ``render``         colours of poses x pixels (rays, coarse and importance samples, composite)
* ``step``           one filter step: weight the particles, resample them, move them
* ``localize``       a whole coarse-to-fine run on the device
* ``map_grad``       loss and gradient of the map's weights at sampled points
* ``proposal_grad``  loss and gradient of the learned proposal sampler

The FP32 form is measured by its blocks (queries, renders, gradients): the weights of a step are
FP64 numbers and resampled indices, which carry any FP32 rounding of the renders on; steps and runs
use the tensor-core forms, in which they are run in practice.

The maps are stand-ins for trained ones: He-normal weights with the weights of frequency 2^k of the
positional encoding scaled by 2^-k (a trained map is smooth at the scale of its finest frequency),
and the density head shifted and scaled to a field that is empty in half of the space.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2406_12202_gb300 as M

NEAR, FAR, ALPHA, TAU = 2.0, 6.0, 0.05, 0.1
# (fan-in, fan-out) of the map's layers in blob order: trunk 1..8, density, feature, RGB hidden, RGB
LAYERS = [(63, 256)] + [(256, 256)] * 4 + [(319, 256)] + [(256, 256)] * 2 + [(256, 1), (256, 256), (283, 128), (128, 3)]
PROPOSAL = [(39, 64), (64, 64), (64, 64), (64, 64), (64, 1)]
EXACT_MOST = 3_000_000   # samples of a render that exact() evaluates


def listed():
    return [
        # a few hundred points of a map looked up between two steps: latency
        {"name": "query_fp32_small", "kind": "query", "precision": "fp32", "n": 1000},
        # a dense look-up (a slice or a grid of a map)
        {"name": "query_fp32_large", "kind": "query", "precision": "fp32", "n": 262144},
        # the same on the tensor-core form, with a ragged count
        {"name": "query_bf16", "kind": "query", "precision": "bf16", "n": 100003},
        # views of 60 poses at the lowest level, ragged in every count
        {"name": "render_fp32_small", "kind": "render", "precision": "fp32", "n": 61, "b": 33, "level": 0,
         "nc": 48, "nf": 80, "side": 400},
        # the full-size sampler of the FP32 form: 600 poses x 64 pixels x (64 + 128) samples
        {"name": "render_fp32_full", "kind": "render", "precision": "fp32", "n": 600, "b": 64, "level": 2,
         "nc": 64, "nf": 128, "side": 400},
        # the smallest step: 32 particles x 8 pixels, coarse samples only
        {"name": "step_bf16_small", "kind": "step", "precision": "bf16", "n": 32, "b": 8, "level": 2,
         "nc": 32, "nf": 0, "side": 100, "proposal": False},
        # the full-size step in both tensor-core forms, and with the learned proposal
        {"name": "step_bf16_full", "kind": "step", "precision": "bf16", "n": 600, "b": 64, "level": 2,
         "nc": 64, "nf": 128, "side": 400, "proposal": False},
        {"name": "step_fp8_full", "kind": "step", "precision": "fp8", "n": 600, "b": 64, "level": 2,
         "nc": 64, "nf": 128, "side": 400, "proposal": False},
        # global localisation of one query: 1500 particles, three levels, 20 iterations
        {"name": "localize_bf16", "kind": "localize", "precision": "bf16", "q": 1, "n": 1500, "iters": 20,
         "nc": 64, "nf": 128, "proposal": False},
        # 16 queries at once with the learned proposal, up to 4000 particles each
        {"name": "localize_fp8_queries", "kind": "localize", "precision": "fp8", "q": 16, "n": 4000, "iters": 12,
         "nc": 32, "nf": 32, "proposal": True},
        # one batch of map fitting
        {"name": "map_grad", "kind": "map_grad", "n": 16384},
        # one batch of proposal training
        {"name": "proposal_grad", "kind": "proposal_grad", "n": 4096, "bins": 64},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["query", "query", "render", "step", "step", "step", "localize", "map_grad", "proposal_grad"])
    if kind == "query":
        return {"kind": kind, "precision": rng.choice(["fp32", "fp32", "bf16", "fp8"]), "n": _log_int(rng, 100, 262144)}
    if kind == "map_grad":
        return {"kind": kind, "n": _log_int(rng, 500, 32768)}
    if kind == "proposal_grad":
        return {"kind": kind, "n": _log_int(rng, 256, 8192), "bins": rng.choice([32, 48, 64, 96])}
    if kind == "localize":
        prop = rng.random() < 0.5
        return {"kind": kind, "precision": rng.choice(["bf16", "fp8"]), "q": rng.randint(1, 8),
                "n": _log_int(rng, 200, 3000), "iters": rng.randint(3, 10), "nc": 32 if prop else rng.choice([32, 64]),
                "nf": rng.choice([32, 64]), "proposal": prop}
    c = {"kind": kind, "precision": "fp32" if kind == "render" else rng.choice(["bf16", "bf16", "fp8"]),
         "n": _log_int(rng, 20, 600), "b": _log_int(rng, 8, 64), "level": rng.randint(0, 2),
         "nc": rng.choice([16, 32, 48, 64]), "nf": rng.choice([0, 32, 64, 100, 128]), "side": rng.choice([100, 200, 400])}
    if kind == "step":
        c["proposal"] = rng.random() < 0.3
    return c


# ---------------------------------------------------------------------------------------- inputs
def _gen(seed, salt):
    return np.random.Generator(np.random.PCG64([int(seed), salt]))


def _gammas(n_freq):
    """Scale of each entry of the positional encoding: 1 for x, 2^-k for the pair of frequency 2^k."""
    return np.concatenate([np.ones(3)] + [np.full(6, 2.0 ** -k) for k in range(n_freq)])


def _pe(x, n_freq):
    parts = [x]
    for k in range(n_freq):
        parts += [torch.sin(x * 2.0 ** k), torch.cos(x * 2.0 ** k)]
    return torch.cat(parts, -1)


def _split(blob, shapes, dtype=torch.float64):
    """The layers (W [out, in], b [out]) of a weight blob."""
    t = torch.as_tensor(blob).cuda().to(dtype)
    out, p = [], 0
    for fi, fo in shapes:
        out.append((t[p:p + fi * fo].view(fo, fi), t[p + fi * fo:p + fi * fo + fo]))
        p += fi * fo + fo
    return out


def _trunk(L, g):
    h = g
    for l in range(8):
        h = torch.relu((torch.cat([h, g], -1) if l == 5 else h) @ L[l][0].T + L[l][1])
    return h


def _mlp(L, x, d):
    """(density before its ReLU, r, g, b) of the map at points x seen along unit directions d."""
    h = _trunk(L, _pe(x, 10))
    f = h @ L[9][0].T + L[9][1]
    hid = torch.relu(torch.cat([f, _pe(d, 4)], -1) @ L[10][0].T + L[10][1])
    return torch.cat([h @ L[8][0].T + L[8][1], torch.sigmoid(hid @ L[11][0].T + L[11][1])], -1)


def _map_weights(seed):
    rng = _gen(seed, 1)
    parts = []
    for i, (fi, fo) in enumerate(LAYERS):
        w = rng.standard_normal((fo, fi)) * math.sqrt(2.0 / fi)
        if i == 0:
            w *= _gammas(10) * 2.0
        if i == 5:
            w[:, 256:] *= _gammas(10)
        parts += [w.reshape(-1), rng.standard_normal(fo) * 0.05]
    blob = np.concatenate(parts).astype(np.float32)
    # density: zero median and a spread of 3 over the space that rays cross
    x = torch.as_tensor(rng.uniform(-5.0, 5.0, size=(4096, 3))).cuda()
    L = _split(blob, LAYERS)
    s = (_trunk(L, _pe(x, 10)) @ L[8][0].T)[:, 0]
    at = sum(fi * fo + fo for fi, fo in LAYERS[:8])
    scale = 3.0 / float(s.std())
    blob[at:at + 256] *= scale
    blob[at + 256] = -scale * float(s.median())
    return blob


def _proposal_weights(seed):
    rng = _gen(seed, 2)
    parts = []
    for i, (fi, fo) in enumerate(PROPOSAL):
        w = rng.standard_normal((fo, fi)) * math.sqrt(2.0 / fi)
        if i == 0:
            w *= _gammas(6) * 2.0
        parts += [w.reshape(-1), np.full(fo, 1.0 if i == 4 else 0.0)]
    return np.concatenate(parts).astype(np.float32)


def _poses(seed, salt, n):
    rng = _gen(seed, salt)
    yaw = rng.uniform(-math.pi, math.pi, n)
    P = np.zeros((n, 3, 4))
    P[:, 0, 0] = P[:, 2, 2] = np.cos(yaw)
    P[:, 0, 2] = np.sin(yaw)
    P[:, 2, 0] = -np.sin(yaw)
    P[:, 1, 1] = 1.0
    P[:, :, 3] = rng.uniform(-1.0, 1.0, (n, 3))
    return torch.as_tensor(P.reshape(n, 12).astype(np.float32)).cuda()


def _image(seed, salt, side):
    rng = _gen(seed, salt)
    y, x = torch.meshgrid(torch.arange(side) / side, torch.arange(side) / side, indexing="ij")
    img = torch.zeros(side, side, 3)
    for c in range(3):
        for _ in range(6):
            kx, ky, ph = rng.uniform(-6, 6), rng.uniform(-6, 6), rng.uniform(0, 2 * math.pi)
            img[..., c] += torch.sin(2 * math.pi * (kx * x + ky * y) + ph)
    return (0.5 + 0.5 * torch.tanh(img / math.sqrt(6))).cuda().contiguous()


def _points(seed, n):
    """Points of the space that rays cross, and unit view directions."""
    rng = _gen(seed, 3)
    d = rng.standard_normal((n, 3))
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    return (torch.as_tensor(rng.uniform(-5.0, 5.0, (n, 3)).astype(np.float32)).cuda(),
            torch.as_tensor(d.astype(np.float32)).cuda())


def _camera(case):
    side = case.get("side", 400)
    f = float(np.float32(1.389 * side))
    return M.intrinsics(f, f, side / 2, side / 2, side, side)


def _pixels(case, seed):
    w = case["side"] * 2 ** case["level"] // 4
    at = _gen(seed, 4).choice(w * w, size=case["b"], replace=False)
    return torch.as_tensor(np.stack([at % w, at // w], 1).astype(np.int32)).cuda()


def _opts(case):
    o = dict(precision=case["precision"], n_coarse=case["nc"], n_fine=case["nf"], near=NEAR, far=FAR, alpha=ALPHA,
             tau=TAU)
    if case.get("proposal"):
        o.update(use_proposal=True, n_proposal=64, n_guided=case["nc"])
    return M.UpdateOptions(**o)


def _schedule(case):
    n, it = case["n"], case["iters"]
    third = max(1, it // 3)
    return M.schedule([0, 1, 2], [16, 32, 64], [n, max(2 * n // 3, 64), max(n // 3, 64)], n_min=64,
                      iter_caps=[third, third, it], refine=[0.0, 0.0, 0.0], iterations=it)


def _samples(case):
    return case["nc"] + case["nf"]


def _counts(case, seed):
    """Initial particle counts of the queries of a run: up to the case's n."""
    n = case["n"]
    return [n] + [int(v) for v in _gen(seed, 6).integers(max(1, n // 4), n + 1, case["q"] - 1)]


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case}
    if kind in ("query", "map_grad"):
        n = case["n"]
        st["map"] = M.Map(_map_weights(seed), max_rays=n, max_samples=2, max_particles=64)
        st["x"], st["d"] = _points(seed, n)
        if kind == "map_grad":
            rng = _gen(seed, 5)
            t = np.concatenate([np.maximum(rng.standard_normal((n, 1)) * 3.0, 0.0), rng.uniform(0, 1, (n, 3))], 1)
            st["target"] = torch.as_tensor(t.astype(np.float32)).cuda()
        return st
    if kind == "proposal_grad":
        n, nb = case["n"], case["bins"]
        st["map"] = M.Map(_map_weights(seed), max_rays=n, max_samples=2, max_particles=64)
        st["map"].proposal_set(_proposal_weights(seed))
        st["o"], d = _points(seed, n)
        st["o"] *= 0.2
        st["d"] = (d * 1.1).contiguous()
        # targets: a surface somewhere along the ray over a floor of weight
        rng = _gen(seed, 7)
        at = rng.uniform(0, nb, (n, 1))
        h = np.exp(-0.5 * ((np.arange(nb) + 0.5 - at) / 2.0) ** 2) + 0.01
        st["hist"] = torch.as_tensor((h / h.sum(1, keepdims=True)).astype(np.float32)).cuda()
        return st
    if kind == "localize":
        sch = _schedule(case)
        q, n = case["q"], case["n"]
        rays = q * max(n * sch.n_pixels[0], max(min(sch.n_cap[s], max(n, 64)) * sch.n_pixels[s] for s in range(3)))
        stride = max(n, 64)
        st["map"] = M.Map(_map_weights(seed), max_rays=rays, max_samples=max(_samples(case), 64),
                          max_particles=q * stride, max_queries=q)
        st["n0"] = _counts(case, seed)
        st["start"] = _poses(seed, 8, q * stride).view(q, stride, 12)
        st["images"] = [_image(seed, 100 + i, 400) for i in range(q)]
        st["particles"] = torch.empty_like(st["start"])
        # one record of 72 bytes per query and iteration (include/mcl.h), the last 8 a time stamp
        st["log"] = torch.zeros(q * case["iters"] * 72, dtype=torch.uint8, device="cuda")
        st["final_n"] = torch.zeros(q, dtype=torch.int32, device="cuda")
        st["schedule"], st["K"], st["opts"] = sch, _camera(case), _opts(case)
        if case["proposal"]:
            st["map"].proposal_set(_proposal_weights(seed))
        return st
    n, b = case["n"], case["b"]
    st["map"] = M.Map(_map_weights(seed), max_rays=n * b, max_samples=max(_samples(case), 64), max_particles=n)
    if case.get("proposal"):
        st["map"].proposal_set(_proposal_weights(seed))
    st["poses"] = _poses(seed, 8, n)
    st["pixels"] = _pixels(case, seed)
    st["K"], st["opts"] = _camera(case), _opts(case)
    if kind == "step":
        st["image"] = _image(seed, 100, case["side"])
        st["u0"] = float(_gen(seed, 9).uniform())
        st["seed"] = int(seed)
    return st


def run(state):
    case, m = state["case"], state["map"]
    kind = case["kind"]
    if kind == "query":
        return m.query(state["x"], state["d"], case["precision"])
    if kind == "render":
        return m.render(state["poses"], state["K"], case["level"], state["pixels"], state["opts"])
    if kind == "step":
        out = m.update(state["poses"], state["image"], state["K"], case["level"], state["pixels"], state["opts"])
        idx = m.resample(out["w"], case["n"], state["u0"])
        moved = M.predict(state["poses"], idx, case["n"], 0.05, 0.05, state["seed"], 1)
        return {"logw": out["logw"], "w": out["w"], "mask": out["mask"], "idx": idx, "poses": moved}
    if kind == "localize":
        state["particles"].copy_(state["start"])
        log, final_n = m.localize(state["particles"], state["n0"], state["images"], state["K"], state["schedule"],
                                  state["opts"], log=state["log"], final_n=state["final_n"])
        rec = log.view(case["q"], case["iters"], 72)
        return {"particles": state["particles"], "final_n": final_n,
                "counts": rec[:, :, :24].contiguous().view(torch.int32),
                "estimates": rec[:, :, 24:64].contiguous().view(torch.float64)}
    if kind == "map_grad":
        return m.loss_grad(state["x"], state["d"], state["target"])
    return m.proposal_loss_grad(state["o"], state["d"], state["hist"], near=NEAR, far=FAR)


# Multiply-accumulates of one sample: the map with its linear feature layer, the proposal.
MAP_MACS = sum(fi * fo for fi, fo in LAYERS)
PROPOSAL_MACS = sum(fi * fo for fi, fo in PROPOSAL)
MAP_BYTES = 4 * sum(fi * fo + fo for fi, fo in LAYERS)
PROPOSAL_BYTES = 4 * sum(fi * fo + fo for fi, fo in PROPOSAL)


def work(case):
    kind = case["kind"]
    if kind == "query":
        return {"bytes": MAP_BYTES + case["n"] * (24 + 16), "flops": 2 * MAP_MACS * case["n"]}
    if kind == "map_grad":
        # forward, gradient of the activations, gradient of the weights
        return {"bytes": 2 * MAP_BYTES + case["n"] * 40, "flops": 6 * MAP_MACS * case["n"]}
    if kind == "proposal_grad":
        rows = case["n"] * case["bins"]
        return {"bytes": 2 * PROPOSAL_BYTES + case["n"] * 24 + rows * 4, "flops": 6 * PROPOSAL_MACS * rows}
    extra = 2 * PROPOSAL_MACS * 64 if case.get("proposal") else 0
    if kind == "localize":
        # every query keeps at least 64 particles; the first iteration has them all
        rays = case["q"] * (case["n"] // 2 * 16 + (case["iters"] - 1) * 64 * 16)
        return {"bytes": MAP_BYTES + case["q"] * (case["n"] * 96 + 400 * 400 * 12),
                "flops": rays * (2 * MAP_MACS * _samples(case) + extra)}
    rays = case["n"] * case["b"]
    bytes_ = MAP_BYTES + case["n"] * 48 + case["b"] * 8 + rays * 12
    if kind == "step":
        bytes_ = MAP_BYTES + case["n"] * (96 + 4 + 8 + 1 + 4) + case["b"] * (8 + 12 * 4 ** (2 - case["level"]))
    return {"bytes": bytes_, "flops": rays * (2 * MAP_MACS * _samples(case) + extra)}


# ------------------------------------------------------------------------------ in 64 bits
def _in_chunks(f, rows, *args, size=131072):
    return torch.cat([f(*(a[i:i + size] for a in args)) for i in range(0, rows, size)])


def _unit(d):
    return d / d.norm(dim=-1, keepdim=True)


def _weights(sigma, z, dn):
    """Eq. 1 weights of samples z [rays, S] with raw densities sigma."""
    delta = torch.cat([(z[:, 1:] - z[:, :-1]) * dn, torch.full_like(z[:, :1], 1e10)], 1)
    a = 1.0 - torch.exp(-torch.relu(sigma) * delta)
    T = torch.cumprod(torch.cat([torch.ones_like(a[:, :1]), 1.0 - a[:, :-1]], 1), 1)
    return T * a


def _importance(w, z, nf):
    """Inverse-CDF samples of the interior weights over the midpoints of z."""
    mid = 0.5 * (z[:, 1:] + z[:, :-1])
    p = w[:, 1:-1] + 1e-5
    cdf = torch.cat([torch.zeros_like(p[:, :1]), torch.cumsum(p / p.sum(1, keepdim=True), 1)], 1)
    u = (torch.arange(nf, dtype=z.dtype, device=z.device) / max(nf - 1, 1)).expand(len(z), nf).contiguous()
    i = torch.searchsorted(cdf.contiguous(), u, right=True)
    lo, hi = (i - 1).clamp(min=0), i.clamp(max=cdf.shape[1] - 1)
    c0, c1 = cdf.gather(1, lo), cdf.gather(1, hi)
    den = torch.where(c1 - c0 < 1e-5, torch.ones_like(c0), c1 - c0)
    return mid.gather(1, lo) + (u - c0) / den * (mid.gather(1, hi) - mid.gather(1, lo))


def _render(case, seed):
    """Colours [rays, 3] of the case's poses x pixels."""
    f64 = torch.float64
    L = _split(_map_weights(seed), LAYERS)
    P = _poses(seed, 8, case["n"]).to(f64).view(-1, 3, 4)
    px = _pixels(case, seed).to(f64)
    s, fac = case["side"], 4 >> case["level"]
    # the level's intrinsics as the library gets them: FP32 numbers over a power of two
    fl, c = float(np.float32(1.389 * s)) / fac, s / 2 / fac
    a = torch.stack([(px[:, 0] + 0.5 - c) / fl, -(px[:, 1] + 0.5 - c) / fl, torch.full_like(px[:, 0], -1.0)], 1)
    d = torch.einsum("nrc,bc->nbr", P[:, :, :3], a).reshape(-1, 3)
    o = P[:, None, :, 3].expand(-1, case["b"], -1).reshape(-1, 3)
    dn, u = d.norm(dim=1, keepdim=True), _unit(d)
    nc, nf = case["nc"], case["nf"]

    def net(z):
        x = (o[:, None] + z[..., None] * d[:, None]).reshape(-1, 3)
        v = u[:, None].expand(-1, z.shape[1], -1).reshape(-1, 3)
        return _in_chunks(lambda x, v: _mlp(L, x, v), len(x), x, v).view(len(z), -1, 4)

    z = (NEAR + (FAR - NEAR) * (torch.arange(nc, dtype=f64, device="cuda") + 0.5) / nc).expand(len(o), nc)
    out = net(z)
    if nf:
        zf = _importance(_weights(out[..., 0], z, dn), z, nf)
        zz, at = torch.sort(torch.cat([z, zf], 1), dim=1, stable=True)
        out, z = torch.cat([out, net(zf)], 1).gather(1, at[..., None].expand(-1, -1, 4)), zz
    w = _weights(out[..., 0], z, dn)
    return (w[..., None] * out[..., 1:]).sum(1)


def exact(case, seed):
    kind = case["kind"]
    if kind == "query":
        L = _split(_map_weights(seed), LAYERS)
        x, d = (t.double() for t in _points(seed, case["n"]))
        return _in_chunks(lambda x, d: _mlp(L, x, _unit(d)), len(x), x, d)
    if kind == "map_grad":
        st = prepare(case, seed)
        L = [(w.clone().requires_grad_(), b.clone().requires_grad_()) for w, b in _split(_map_weights(seed), LAYERS)]
        out = _mlp(L, st["x"].double(), _unit(st["d"].double()))
        t = st["target"].double()
        loss = (1e-2 * (out[:, 0] - t[:, 0]) ** 2 + ((out[:, 1:] - t[:, 1:]) ** 2).sum(1)).mean()
        g = torch.autograd.grad(loss, [p for layer in L for p in layer])
        return float(loss), torch.cat([v.reshape(-1) for v in g])
    if kind == "proposal_grad":
        st = prepare(case, seed)
        n, nb = case["n"], case["bins"]
        L = [(w.clone().requires_grad_(), b.clone().requires_grad_())
             for w, b in _split(_proposal_weights(seed), PROPOSAL)]
        o, d, hist = st["o"].double(), st["d"].double(), st["hist"].double()
        z = (NEAR + (FAR - NEAR) * (torch.arange(nb, dtype=torch.float64, device="cuda") + 0.5) / nb).expand(n, nb)
        h = _pe(o[:, None] + z[..., None] * d[:, None], 6)
        for w, b in L[:4]:
            h = torch.relu(h @ w.T + b)
        w = _weights((h @ L[4][0].T + L[4][1])[..., 0], z, d.norm(dim=1, keepdim=True))
        W = w.sum(1, keepdim=True)
        p = torch.where(W > 0, w / torch.where(W > 0, W, torch.ones_like(W)), torch.zeros_like(w))
        loss = -(hist * torch.log(p + 1e-8)).sum(1).mean()
        g = torch.autograd.grad(loss, [v for layer in L for v in layer])
        return float(loss), torch.cat([v.reshape(-1) for v in g])
    # steps and runs: the last interval of a ray is 1e10 long, so the sign of its last density, which
    # the operands' rounding in 16 or 8 bits decides for some rays, moves a particle's loss at will
    if kind != "render" or case["n"] * case["b"] * _samples(case) > EXACT_MOST:
        return None
    return _render(case, seed)
