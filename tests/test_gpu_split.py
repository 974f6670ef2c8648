"""FP32 form on FP16 operand pairs (csrc/mlp_split.cu): point queries against
the FP64 oracle at the edges of the kernel's units (256 rows, 128 per CTA) and
of its persistent grid, on a dense map, and on a map of copies, which the
dispatch leaves on the SIMT kernels.

Tolerance: an FP32 FMA chain of 256 terms rounds by about sqrt(256) 2^-24 =
9.5e-7 of its result; nine layers in a row add up to 8.6e-6 of the largest
outputs (the pairs are held to the chain they replace)."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import synth
from gpu_helpers import lib

pytestmark = pytest.mark.gpu

TOL = 9 * np.sqrt(256) * 2.0 ** -24


def _points(n, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    x = rng.uniform(-2.9, 2.9, size=(n, 3))
    d = rng.normal(size=(n, 3))
    return x.astype(np.float32), (d / np.linalg.norm(d, axis=1, keepdims=True)).astype(np.float32)


@pytest.mark.parametrize("blob", ["dense", "copies"])
@pytest.mark.parametrize("n", [1, 127, 129, 255, 257, 76 * 256 + 1])
def test_query_against_oracle(n, blob):
    import torch
    M = lib()
    w = synth.he_init_weights(2, bias_std=0.1) if blob == "dense" else synth.room_map_weights(0)[0]
    x, d = _points(n, n)
    gm = M.Map(w, max_rays=n, max_samples=2, max_particles=8)
    try:
        got = gm.query(torch.tensor(x, device="cuda"), torch.tensor(d, device="cuda"), "fp32")
        got = got.cpu().numpy().astype(np.float64)
        assert gm.read_status()[0] == 0
    finally:
        gm.close()
    at = np.unique(np.r_[np.arange(min(n, 300)), np.arange(max(0, n - 300), n)])
    dh = d[at].astype(np.float64)
    sig, rgb = oracle.mlp(w, x[at].astype(np.float64), dh / np.linalg.norm(dh, axis=1, keepdims=True))
    ref = np.c_[sig, rgb]
    err = np.abs(got[at] - ref)
    big = np.maximum(np.abs(ref).max(0), 1e-3)
    assert np.all(err <= TOL * big), (err / big).max()


def test_huge_and_non_finite_points():
    """Points far outside any scene keep finite rows finite, and a NaN point
    stays in its own row."""
    import torch
    M = lib()
    w = synth.he_init_weights(2, bias_std=0.1)
    x, d = _points(300, 5)
    gm = M.Map(w, max_rays=300, max_samples=2, max_particles=8)
    try:
        q = lambda v: gm.query(torch.tensor(v, device="cuda"), torch.tensor(d, device="cuda"), "fp32").cpu().numpy()
        ref = q(x)
        y = x.copy()
        y[7] = [np.nan, 0.0, 0.0]
        y[200] = [np.inf, 1.0, 2.0]
        y[31] = [1e20, -3.0, 2.0]
        got = q(y)
        keep = np.ones(300, bool)
        keep[[7, 31, 200]] = False
        assert np.array_equal(got[keep], ref[keep])
        assert np.isfinite(got[31]).all()
    finally:
        gm.close()
