"""Kernels that share work among lanes, warps and CTAs, at the sizes where
their split changes: pixel sets (a warp), weights (one to eight CTAs), composites (rings of 16 samples) and
the map's gradient (chunks of 1,024 rows, tiles of 128 and 64)."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import synth
from gpu_helpers import lib

pytestmark = pytest.mark.gpu


def _poses(n, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    yaw = rng.uniform(-3, 3, n)
    p = np.zeros((n, 3, 4))
    p[:, 0, 0] = p[:, 2, 2] = np.cos(yaw)
    p[:, 0, 2], p[:, 2, 0], p[:, 1, 1] = np.sin(yaw), -np.sin(yaw), 1.0
    p[:, :, 3] = rng.uniform(-1, 1, (n, 3))
    return p.reshape(n, 12).astype(np.float32)


@pytest.mark.parametrize("W,H,B", [(1, 1, 1), (8, 8, 64), (7, 5, 33), (100, 100, 31), (400, 400, 256), (40, 30, 1024)])
def test_pixel_set(W, H, B):
    got = lib().draw_pixels(W, H, B, 11, 5).cpu().numpy()
    assert np.array_equal(got, oracle.pixel_set(W, H, B, 11, 5))


@pytest.mark.parametrize("n", [1, 32, 33, 64, 65, 128, 129, 1024, 1025, 2500])
def test_weights(n):
    """log w within some ulps of FP64 at |log w| < 300, so w within 1e-12."""
    import torch
    M = lib()
    gm = M.Map(synth.he_init_weights(2, bias_std=0.1), max_rays=3 * n, max_samples=2, max_particles=n)
    P = _poses(n, 1)
    if n > 40:
        P[n - 3, 3] = np.nan                     # no weight
    K = M.intrinsics(30.0, 30.0, 8.0, 8.0, 16, 16)
    try:
        r = gm.update(torch.tensor(P, device="cuda"), torch.rand(16, 16, 3, device="cuda"), K, 2,
                      torch.tensor([[1, 2], [9, 4], [3, 15]], dtype=torch.int32, device="cuda"),
                      M.UpdateOptions(n_coarse=2, n_fine=0), debug=True)
        S, w, mask, logw = (r[k].cpu().numpy() for k in ("S", "w", "mask", "logw"))
        assert gm.read_status()[1] == (1 if n > 40 else 0)
    finally:
        gm.close()
    with np.errstate(invalid="ignore"):
        l = np.where(np.isfinite(S), 4 * (np.log(3.0) - np.log(np.maximum(S.astype(np.float64), 1e-30))), -np.inf)
    ref = np.exp(l - l.max())
    ref /= ref.sum()
    assert np.all(np.abs(w - ref) <= 1e-12 * ref)
    assert np.array_equal(logw, l.astype(np.float32)) or np.allclose(logw, l, rtol=2.0 ** -23)
    assert np.array_equal(mask != 0, (ref >= 1e-3 / n) & (ref > 0))


@pytest.mark.parametrize("nc", [2, 7, 8, 9, 16, 17, 33, 256])
def test_composite(nc):
    """Rays of a whole warp and one more; colours against the FP64 oracle, to
    the FP32 bar of renders (1e-4 relative)."""
    import torch
    M = lib()
    blob = synth.he_init_weights(2, bias_std=0.1)
    P = _poses(11, 5)
    px = np.array([[1, 2], [9, 4], [3, 15]], dtype=np.int32)
    K4 = (30.0, 30.0, 8.0, 8.0)
    gm = M.Map(blob, max_rays=33, max_samples=256, max_particles=16)
    try:
        rgb = gm.render(torch.tensor(P, device="cuda"), M.intrinsics(*K4, 16, 16), 2, torch.tensor(px, device="cuda"),
                        M.UpdateOptions(n_coarse=nc, n_fine=0))
        rgb = (rgb[0] if isinstance(rgb, tuple) else rgb).cpu().numpy().reshape(33, 3)
    finally:
        gm.close()
    o, d = zip(*[oracle.ray(p.astype(np.float64), *K4, int(u), int(v)) for p in P for u, v in px])
    ref = oracle.render_rays(blob, np.array(o), np.array(d), oracle.make_opts(n_coarse=nc, n_fine=0))
    ref = np.asarray(ref["rgb"] if isinstance(ref, dict) else ref[0]).reshape(33, 3)
    assert np.all(np.abs(rgb - ref) <= 1e-4 * np.maximum(np.abs(ref), 1.0))


LAYERS = [(63, 256)] + [(256, 256)] * 4 + [(319, 256)] + [(256, 256)] * 2 + [(256, 1), (256, 256), (283, 128), (128, 3)]


def _pe(x, n):
    import torch
    return torch.cat([x] + [f(x * 2.0 ** k) for k in range(n) for f in (torch.sin, torch.cos)], -1)


@pytest.mark.parametrize("n", [1, 127, 129, 1023, 1025, 2049])
def test_map_gradient(n):
    """Against FP64 autograd, per tensor: roundings of 18 chained layers are
    about 2e-5 of a gradient's norm; a ReLU input within FP32 of zero (a few
    of the 2,176 n) moves it by one unit of one row, 1 / sqrt(256 n) of it, and
    a lost row would by 1 / sqrt(n)."""
    import torch
    M = lib()
    blob = synth.he_init_weights(4, bias_std=0.05)
    x, d = synth.room_fit_points(n, n)
    rng = np.random.Generator(np.random.PCG64(n))
    t = rng.uniform(0, 1, (n, 4)).astype(np.float32)
    gm = M.Map(blob, max_rays=max(n, 64))
    try:
        loss, g = gm.loss_grad(*(torch.tensor(a, device="cuda") for a in (x, d, t)), sigma_weight=1e-2)
        g = g.cpu().double()
    finally:
        gm.close()
    p = torch.tensor(blob, dtype=torch.float64, requires_grad=True)
    L, at = [], 0
    for fi, fo in LAYERS:
        L.append((p[at:at + fi * fo].view(fo, fi), p[at + fi * fo:at + fi * fo + fo]))
        at += fi * fo + fo
    X, D, T = (torch.tensor(a, dtype=torch.float64) for a in (x, d, t))
    e = _pe(X, 10)
    h = e
    for l in range(8):
        h = torch.relu((torch.cat([h, e], -1) if l == 5 else h) @ L[l][0].T + L[l][1])
    f = h @ L[9][0].T + L[9][1]
    hid = torch.relu(torch.cat([f, _pe(D / D.norm(dim=1, keepdim=True), 4)], -1) @ L[10][0].T + L[10][1])
    out = torch.cat([h @ L[8][0].T + L[8][1], torch.sigmoid(hid @ L[11][0].T + L[11][1])], -1)
    ref = ((out - T) ** 2 * torch.tensor([1e-2, 1.0, 1.0, 1.0])).sum(1).mean()
    ref.backward()
    assert abs(loss - ref.item()) <= 1e-5 * ref.item()
    tol = 2e-5 + 4 / np.sqrt(256.0 * n)
    at = 0
    for fi, fo in LAYERS:
        for m in (fi * fo, fo):
            a, b = g[at:at + m], p.grad[at:at + m]
            assert (a - b).norm() <= min(tol, 0.5 / np.sqrt(n)) * b.norm(), (at, (a - b).norm() / b.norm())
            at += m
