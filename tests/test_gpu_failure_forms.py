"""As test_gpu_failure.py, for every kernel that calls run on without tuning: the
FP32 form's CTA-pair kernel, the BF16 pair and the FP8 kernel, in their versions
for point queries and for rays, with one and with several units of rows per
CTA (or pair).  The held weight stream issues no copy, so the waits of the
relay, gate, epilogue and encoding warps run out at 2 ms; the kernels stop,
give their tensor memory back and report, and the next call gives the same
results as before."""
import time

import numpy as np
import pytest

import synth
from gpu_helpers import lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("call", ["query", "query, several units", "render"])
@pytest.mark.parametrize("precision", ["fp32", "bf16", "fp8"])
def test_held_launch_of_the_untuned_kernels(precision, call):
    import torch
    M = lib()
    gm = M.Map(synth.he_init_weights(0), max_rays=100_000, max_samples=32, max_particles=2048)
    try:
        rng = np.random.default_rng(11)
        if call == "render":
            P = torch.tensor(synth.random_particles(3, 200)[0], dtype=torch.float32, device="cuda")
            px = torch.tensor(synth.pixel_set(3, 100, 100, 16), dtype=torch.int32, device="cuda")
            K = M.intrinsics(138.9, 138.9, 50.0, 50.0, 100, 100)
            o = M.UpdateOptions(n_coarse=32, n_fine=0, precision=precision)
            run = lambda: gm.render(P, K, 2, px, o)
        else:
            n = 3000 if call == "query" else 100_000
            x = torch.tensor(rng.uniform(-1.5, 1.5, size=(n, 3)), dtype=torch.float32, device="cuda")
            d = torch.tensor(rng.normal(size=(n, 3)), dtype=torch.float32, device="cuda")
            run = lambda: gm.query(x, d, precision)
        ref = run().clone()
        torch.cuda.synchronize()
        assert gm.read_status()[0] == M.MCL_OK
        gm.inject_weight_stall(1, 2.0)
        t0 = time.perf_counter()
        run()
        torch.cuda.synchronize()
        waited = time.perf_counter() - t0
        assert gm.read_status()[0] == M.MCL_ERR_TIMEOUT
        assert waited < 1.0
        again = run()
        torch.cuda.synchronize()
        assert gm.read_status()[0] == M.MCL_OK
        assert torch.equal(again, ref)
    finally:
        gm.close()
