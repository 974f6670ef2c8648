"""FP32 form on FP16 operand pairs: the scale of each point's encoding travels
beside its operand, from the warp that encodes to the warps that add the
products.  Points whose scales differ from row to row, over several units per
CTA pair, must not depend on where in the call they stand."""
from __future__ import annotations

import numpy as np
import pytest

import synth
from gpu_helpers import lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [300, 76 * 256 + 1, 3 * 76 * 256 + 57])
def test_points_do_not_depend_on_their_place(n):
    import torch
    M = lib()
    rng = np.random.Generator(np.random.PCG64(n))
    # encodings scaled by 2^13 down to 2^3
    x = rng.uniform(-1, 1, (n, 3)) * 2.0 ** rng.integers(0, 11, (n, 1))
    d = rng.normal(size=(n, 3))
    gm = M.Map(synth.he_init_weights(2, bias_std=0.1), max_rays=n, max_samples=2, max_particles=8)
    try:
        xt, dt = (torch.tensor(a, dtype=torch.float32, device="cuda") for a in (x, d))
        ref = gm.query(xt, dt, "fp32")
        assert bool(torch.isfinite(ref).all())
        for shift in (1, 128, 256 * 76 + 3):
            p = torch.roll(torch.randperm(n, generator=torch.Generator().manual_seed(shift)), shift).cuda()
            got = gm.query(xt[p].contiguous(), dt[p].contiguous(), "fp32")
            assert torch.equal(got, ref[p])
        assert gm.read_status()[0] == M.MCL_OK
    finally:
        gm.close()
