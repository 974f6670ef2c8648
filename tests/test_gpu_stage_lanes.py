"""The stages that a warp does for 32 rays or eight particles together, at the
sizes where a warp is partly filled, a ring wraps or one list of a merge runs
dry: a ray's or a particle's result must not depend on its neighbours, and is
held to the oracle."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import synth
from gpu_helpers import lib

pytestmark = pytest.mark.gpu

K4 = (30.0, 30.0, 8.0, 8.0)
PX = np.array([[1, 2], [9, 4], [3, 15]], dtype=np.int32)


def _smooth_map():
    """A dense map whose weights of frequency 2^k are scaled by 2^-k, so that the
    FP32 rounding of a sample's place moves no colour by more than FP32 does."""
    blob = synth.he_init_weights(2, bias_std=0.1)
    g = np.concatenate([np.ones(3)] + [np.full(6, 2.0 ** -k) for k in range(10)]).astype(np.float32)
    for name, cols in (("trunk1", slice(0, 63)), ("trunk6", slice(256, 319))):
        ow, ob, fi, fo = synth.blob_offsets()[name]
        blob[ow:ob].reshape(fo, fi)[:, cols] *= g
    return blob


def _poses(n, seed):
    return synth.random_particles(seed, n)[0].astype(np.float32)


@pytest.mark.parametrize("scene", ["smooth", "wall"])
@pytest.mark.parametrize("nc,nf", [(2, 1), (3, 2), (7, 33), (17, 16), (16, 100), (256, 128), (256, 256)])
def test_rays_of_a_warp(nc, nf, scene):
    """33 rays (a warp and one) of 11 poses: colours to the FP32 bar of renders
    (1e-4 relative), and the same bits with the poses in reverse and one by one.
    wall: a room whose wall a few samples of one coarse interval see, so that
    nearly all importance samples fall between two coarse ones."""
    import torch
    M = lib()
    blob = _smooth_map() if scene == "smooth" else synth.room_map_weights(0)[0]
    P = _poses(11, 5)
    gm = M.Map(blob, max_rays=33, max_samples=512, max_particles=16)
    try:
        K, px, o = M.intrinsics(*K4, 16, 16), torch.tensor(PX, device="cuda"), M.UpdateOptions(n_coarse=nc, n_fine=nf)
        f = lambda Q: gm.render(torch.tensor(Q, device="cuda"), K, 2, px, o).reshape(-1, 3, 3).cpu().numpy()
        rgb = f(P)
        assert np.array_equal(rgb, f(np.ascontiguousarray(P[::-1]))[::-1])
        assert np.array_equal(rgb, np.concatenate([f(P[i:i + 1]) for i in range(11)]))
    finally:
        gm.close()
    od, dd = zip(*[oracle.ray(p.astype(np.float64), *K4, int(u), int(v)) for p in P for u, v in PX])
    ref = oracle.render_rays(blob, np.array(od), np.array(dd), oracle.make_opts(n_coarse=nc, n_fine=nf))
    ref = np.asarray(ref["rgb"] if isinstance(ref, dict) else ref[0]).reshape(11, 3, 3)
    assert np.all(np.abs(rgb - ref) <= 1e-4 * np.maximum(np.abs(ref), 1.0))


@pytest.mark.parametrize("n", [1, 7, 8, 9, 33])
def test_prediction_of_partly_filled_warps(n):
    """Particle k draws from its own part of the stream whatever n is; indices
    outside the set give NaN poses and leave their neighbours alone.  Sigmas that
    FP32 holds exactly; bar as in test_gpu_parity.py."""
    import torch
    M = lib()
    P = _poses(12, 8)
    idx = np.random.default_rng(n).integers(0, 12, n).astype(np.int32)
    bad = idx.copy()
    bad[::3], bad[1::5] = -1, 12
    at = lambda v: M.predict(torch.tensor(P, device="cuda"), torch.tensor(v, device="cuda"), n, 0.0625, 0.03125, 77,
                             3).cpu().numpy()
    out, holes = at(idx), at(bad)
    keep = bad == idx
    assert np.array_equal(holes[keep], out[keep]) and np.isnan(holes[~keep]).all()
    more = M.predict(torch.tensor(P, device="cuda"), torch.tensor(np.r_[idx, idx], device="cuda"), 2 * n, 0.0625,
                     0.03125, 77, 3).cpu().numpy()
    assert np.array_equal(more[:n], out)
    ref = oracle.predict(P.astype(np.float64)[idx], oracle.motion_noise(n, 77, 3, 0.0625, 0.03125))
    assert np.allclose(out, ref.reshape(n, 12), rtol=0, atol=3e-6)
