"""Training entry points on a stream of the caller's that is not ordered with
the default stream (torch's side streams are non-blocking)."""
from __future__ import annotations

import numpy as np
import pytest

import synth
from gpu_helpers import lib

pytestmark = pytest.mark.gpu


def test_fit_on_a_side_stream_behind_a_busy_default_stream():
    """Every step of a fit, the clearing of Adam's moments included, runs on the
    caller's stream: with work queued on the default stream, and on a map whose
    scratch holds the values of an earlier call, the fit gives the bits of a
    first one (fits are deterministic)."""
    import torch
    M = lib()
    n = 3000
    x, d = synth.room_fit_points(3, n)
    sig, rgb = synth.room_field(x)
    t = np.concatenate([sig[:, None], rgb], 1).astype(np.float32)
    xt, dt, tt = (torch.tensor(a, device="cuda") for a in (x, d, t))
    blob = synth.he_init_weights(5, bias_std=0.05)
    cfg = dict(steps=12, batch=1000, lr=1e-3, lr_end=1e-3, sigma_weight=1e-2, seed=3)
    first, again = M.Map(blob, max_rays=4096), M.Map(blob, max_rays=4096)
    try:
        log0 = first.fit(xt, dt, tt, **cfg)
        w0 = first.weights()
        # fills the scratch (gradients do not change the map)
        again.loss_grad(xt, dt, tt * 3.0 + 1.0)
        side = torch.cuda.Stream()
        torch.cuda.synchronize()
        torch.cuda._sleep(200_000_000)           # about 0.1 s on the default stream
        with torch.cuda.stream(side):
            log1 = again.fit(xt, dt, tt, **cfg)
        torch.cuda.synchronize()
        assert torch.equal(log0, log1)
        assert np.array_equal(w0, again.weights())
    finally:
        first.close()
        again.close()
