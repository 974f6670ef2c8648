"""The device loop in FP32 on a dense map: its MLP runs on operand pairs with the
number of rows in device memory (CTA pairs beyond them have no unit), and the
densities of a first pass come from the SIMT kernels.  Every record has to follow
from single FP32 updates of the same particles, as the BF16 runs of
test_gpu_loop.py do."""
import numpy as np
import pytest

import oracle
import synth
from gpu_helpers import lib

pytestmark = pytest.mark.gpu

SIDE, F = 100, 138.9


@pytest.mark.parametrize("nc,nf", [(32, 32), (24, 0)])
def test_records_follow_from_single_updates(nc, nf):
    import torch
    M = lib()
    Q, stride, iters = 2, 150, 4
    n0 = [150, 70]
    levels, pixels, caps, n_min = [1, 2], [12, 24], [150, 60], 16
    refine, iter_caps = [0.0, 0.0], [2, 10]
    seed = 77
    K = M.intrinsics(F, F, SIDE / 2, SIDE / 2, SIDE, SIDE)
    opts = M.UpdateOptions(n_coarse=nc, n_fine=nf, precision="fp32", seed=seed)
    # far more rays than the later iterations have
    gm = M.Map(synth.he_init_weights(2, bias_std=0.1), max_rays=20000, max_samples=64, max_particles=Q * stride,
               max_queries=Q)
    try:
        imgs = [torch.tensor(synth.smooth_image(20 + q, SIDE, SIDE), dtype=torch.float32, device="cuda") for q in range(Q)]
        parts = torch.full((Q, stride, 12), float("nan"), device="cuda")
        for q in range(Q):
            parts[q, :n0[q]] = torch.tensor(synth.random_particles(30 + q, n0[q])[0], dtype=torch.float32, device="cuda")

        def run(t, graph=False):
            p = parts.clone()
            sch = M.schedule(levels, pixels, caps, n_min=n_min, iter_caps=iter_caps, refine=refine, iterations=t)
            log, fin = gm.localize(p, n0, imgs, K, sch, opts, use_graph=graph)
            return p, M.Map.decode_log(log, Q, t), [int(v) for v in fin.cpu()]

        runs = [None] + [run(t) for t in range(1, iters + 1)]
        p_all, recs, fin = runs[iters]
        for q in range(Q):
            stage, it = 0, 0
            Pq = parts[q, :n0[q]]
            for t in range(iters):
                r, B, lev = recs[q][t], pixels[stage], levels[stage]
                f = 4 >> lev
                assert r["stage"] == stage and r["n_particles"] == len(Pq) and r["status"] == 0
                c = (q << 32) | (t << 2)
                px = M.draw_pixels(SIDE // f, SIDE // f, B, seed, c)
                out = gm.update(Pq.contiguous(), imgs[q], K, lev, px, opts)
                st = oracle.loop_statistics(Pq.cpu().numpy().astype(np.float64), out["w"].cpu().numpy(),
                                            out["mask"].cpu().numpy())
                assert r["n_survivors"] == st["n_survivors"]
                assert r["spread"] == pytest.approx(st["spread"], rel=1e-9)
                assert np.allclose(r["est"][:3], st["mean"], rtol=0, atol=1e-12)
                stage, it, n_next = oracle.loop_schedule(stage, it, st["n_survivors"], st["spread"], refine, iter_caps,
                                                         caps, n_min, stride)
                # the particles of the next iteration, to the bit
                idx = gm.resample(out["w"], n_next, oracle.uniform(seed, c + 1, 0))
                nxt = M.predict(Pq.contiguous(), idx, n_next, 0.05, 0.05, seed, c + 2)
                assert runs[t + 1][2][q] == n_next
                assert torch.equal(runs[t + 1][0][q, :n_next], nxt)
                Pq = nxt
        g_p, g_recs, g_fin = run(iters, graph=True)
        assert g_fin == fin
        for q in range(Q):
            assert torch.equal(g_p[q, :fin[q]], p_all[q, :fin[q]])
        assert gm.read_status()[0] == M.MCL_OK
    finally:
        gm.close()
