"""Device memory of the training and gradient entry points: training runs give
theirs back before they return, gradient calls leave at most 1 GiB with the map."""
from __future__ import annotations

import numpy as np
import pytest

import synth
from gpu_helpers import lib

pytestmark = pytest.mark.gpu

MIB = 1 << 20


def _free():
    import torch
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


def _room_points(n):
    import torch
    x, d = synth.room_fit_points(3, n)
    sig, rgb = synth.room_field(x)
    t = np.concatenate([sig[:, None], rgb], 1).astype(np.float32)
    return [torch.tensor(a, device="cuda") for a in (x, d, t)]


def test_training_runs_give_their_scratch_back():
    """A fit's batch of 16,384 points takes some 230 MiB, a training batch of
    4,096 rays x 64 bins some 650; the margin is what the driver and the caching
    allocator keep.  A small run first: the driver keeps some 94 MiB for the
    training kernels from their first launch on, whatever the batch."""
    import torch
    M = lib()
    gm = M.Map(synth.he_init_weights(0), max_rays=4096, max_samples=64)
    try:
        pts = _room_points(16384)
        gm.fit(*_room_points(64), steps=1, batch=64)      # kernels loaded
        before = _free()
        gm.fit(*pts, steps=2, batch=16384)
        assert _free() >= before - 64 * MIB
        gm.proposal_set(synth.proposal_init_weights(0))
        P = torch.tensor(synth.random_particles(3, 128)[0], dtype=torch.float32, device="cuda")
        px = torch.tensor(synth.pixel_set(3, 100, 100, 32), dtype=torch.int32, device="cuda")
        K = M.intrinsics(138.9, 138.9, 50.0, 50.0, 100, 100)
        o = M.UpdateOptions(n_coarse=16, n_fine=16)
        gm.proposal_train(P, px, K, 2, o, epochs=1, batch_rays=64, n_bins=64)
        before = _free()
        gm.proposal_train(P, px, K, 2, o, epochs=1, batch_rays=4096, n_bins=64)
        assert _free() >= before - 64 * MIB
    finally:
        gm.close()


def test_gradient_calls_keep_a_bounded_block_until_the_map_is_closed():
    M = lib()
    start = None
    gm = M.Map(synth.he_init_weights(0), max_rays=4096)
    try:
        gm.loss_grad(*_room_points(64))                   # kernels loaded
        pts = _room_points(16384)
        big = _room_points(100_000)                       # about 1.4 GB of scratch
        start = _free()
        g = gm.loss_grad(*pts)[1]
        kept = start - _free()
        assert 100 * MIB <= kept <= 1024 * MIB + 64 * MIB
        assert bool((gm.loss_grad(*pts)[1] == g).all()) and start - _free() <= kept + 64 * MIB
        gm.loss_grad(*big)
        assert start - _free() <= 1024 * MIB + 64 * MIB
        # a training run of the same map uses the kept block
        gm.fit(*pts, steps=1, batch=8192)
        assert start - _free() <= 1024 * MIB + 64 * MIB
    finally:
        gm.close()
    assert _free() >= start - 64 * MIB
