"""Which maps the FP32 form runs on FP16 operand pairs (csrc/mlp_split.cu): only
those whose every row is a sum of many terms, and there the pairs are no further
from FP64 than the FMA chain they replace.

The chain's own error comes from a twin of the map: one unit of the first layer
that nothing reads holds a single weight instead of a dense row, which changes
no output and sends the twin to the SIMT kernels.  The route shows in the number
of kernels a query launches: three (set-up, per-point bias, the fused MLP)."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import synth
from gpu_helpers import lib

pytestmark = pytest.mark.gpu


def _layer(blob, name):
    """(W [out, in], b [out]) of a layer, views into the blob."""
    ow, ob, fi, fo = synth.blob_offsets()[name]
    return blob[ow:ob].reshape(fo, fi), blob[ob:ob + fo]


def _dense(seed, decay=False):
    blob = synth.he_init_weights(seed, bias_std=0.1)
    if decay:      # weights of frequency 2^k scaled by 2^-k, as of a smooth map
        g = np.concatenate([np.ones(3)] + [np.full(6, 2.0 ** -k) for k in range(10)])
        _layer(blob, "trunk1")[0][:] *= g.astype(np.float32)
        _layer(blob, "trunk6")[0][:, 256:] *= g.astype(np.float32)
    _layer(blob, "trunk2")[0][:, 255] = 0.0      # nothing reads unit 255 of trunk1
    return blob


def _twin(blob):
    blob = blob.copy()
    _layer(blob, "trunk1")[0][255, 1:] = 0.0
    return blob


def _thin(name, k, rows):
    """A dense map whose given rows of one layer hold k equal weights."""
    blob = _dense(2)
    W = _layer(blob, name)[0]
    rng = np.random.Generator(np.random.PCG64(k))
    for o in rows:
        at = rng.permutation(W.shape[1])[:k]
        v = rng.choice([-1.0, 1.0], k) * np.sqrt(2.0 / k)
        W[o] = 0.0
        W[o, at] = v
    return blob


def _room_beside_dense():
    """The room map (units 0..55, rows of one to four terms) with its idle units
    filled by a dense network that the density never reads."""
    blob = synth.room_map_weights(0)[0]
    fill = synth.he_init_weights(9, bias_std=0.1)
    for l in range(1, 9):
        W, b = _layer(blob, f"trunk{l}")
        F, c = _layer(fill, f"trunk{l}")
        b[56:] = c[56:]
        if l == 1:
            W[56:] = F[56:]
        else:
            W[56:, 56:] = F[56:, 56:]
    return blob


def _points(n, seed):
    x, d = synth.room_fit_points(seed, n)
    return x, d


def _query(M, blob, x, d):
    """The FP32 query and the number of kernels it launched."""
    import torch
    gm = M.Map(blob, max_rays=len(x), max_samples=2, max_particles=8)
    try:
        xt, dt = torch.tensor(x, device="cuda"), torch.tensor(d, device="cuda")
        before = gm.profile_read()[1]
        out = gm.query(xt, dt, "fp32")
        launched = gm.profile_read()[1] - before
        return out.cpu().numpy().astype(np.float64), launched
    finally:
        gm.close()


def _exact(blob, x, d):
    dh = d.astype(np.float64)
    sig, rgb = oracle.mlp(blob, x.astype(np.float64), dh / np.linalg.norm(dh, axis=1, keepdims=True))
    return np.c_[sig, rgb]


MAPS = {
    "dense": (lambda: _dense(2), True),
    "dense, smooth": (lambda: _dense(3, decay=True), True),
    "first layer: 32 of 63": (lambda: _thin("trunk1", 32, range(256)), True),
    "trunk5: 128 of 256": (lambda: _thin("trunk5", 128, range(256)), True),
    "twin": (lambda: _twin(_dense(2)), False),
    "first layer: 16 of 63 in one row": (lambda: _thin("trunk1", 16, [3]), False),
    "trunk5: 64 of 256 in one row": (lambda: _thin("trunk5", 64, [7]), False),
    "trunk5: copies in eight rows": (lambda: _thin("trunk5", 1, range(8)), False),
    "density head: one term": (lambda: _thin("sigma", 1, [0]), False),
    "room beside a dense network": (_room_beside_dense, False),
}


@pytest.mark.parametrize("name", MAPS)
def test_route(name):
    """Tolerance as in test_gpu_split.py, nine FP32 chains of 256 terms; for the
    room, whose density is 64 (64 m - 192) behind the wall at m = 3, four
    roundings of FP32 numbers between 128 and 256 (2^-17 each) before the slope
    of 64, over the largest density of 64."""
    M = lib()
    make, pairs = MAPS[name]
    tol = 4 * 2.0 ** -17 if "room" in name else 9 * np.sqrt(256) * 2.0 ** -24
    blob = make()
    x, d = _points(700, 1)
    got, launched = _query(M, blob, x, d)
    ref = _exact(blob, x, d)
    err = np.abs(got - ref) / np.maximum(np.abs(ref).max(0), 1e-3)
    assert np.all(err <= tol), err.max()
    assert (launched == 3) == pairs, launched


@pytest.mark.parametrize("seed,decay", [(2, False), (4, False), (11, False), (3, True), (5, True)])
def test_pairs_are_no_further_from_fp64_than_the_chain(seed, decay):
    M = lib()
    blob = _dense(seed, decay)
    x, d = _points(6000, seed)
    ref = _exact(blob, x, d)
    pairs, launched = _query(M, blob, x, d)
    chain, launched_chain = _query(M, _twin(blob), x, d)
    assert launched == 3 and launched_chain > 3
    e, c = np.abs(pairs - ref), np.abs(chain - ref)
    for col in (slice(0, 1), slice(1, 4)):
        assert np.sqrt((e[:, col] ** 2).mean()) <= np.sqrt((c[:, col] ** 2).mean())
        assert e[:, col].max() <= c[:, col].max()


def test_maps_on_the_simt_kernels_launch_those_alone():
    """Encoding, nine trunk and feature layers, two RGB layers and the density
    head are 13 launches; a query adds its set-up, a render without importance
    samples its rays and its composite.  The per-ray bias is the pairs'."""
    import torch
    M = lib()
    blob = _twin(_dense(2))
    x, d = _points(700, 1)
    assert _query(M, blob, x, d)[1] == 1 + 13
    gm = M.Map(blob, max_rays=64, max_samples=16, max_particles=8)
    try:
        P = torch.tensor(synth.random_particles(3, 8)[0], dtype=torch.float32, device="cuda")
        px = torch.tensor([[1, 2], [9, 4], [3, 15]], dtype=torch.int32, device="cuda")
        before = gm.profile_read()[1]
        gm.render(P, M.intrinsics(30.0, 30.0, 8.0, 8.0, 16, 16), 2, px, M.UpdateOptions(n_coarse=16, n_fine=0))
        assert gm.profile_read()[1] - before == 2 + 13
    finally:
        gm.close()
