"""Batches of few blocks (tile kernels) and of many (block kernels), against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_util import TOL, rel_err_per_m, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built(cuda_device):
    from paper_2408_16847_gb300 import build
    build()


def _run(sizes, reach):
    """sizes: (nside, bins, m_max) of the members.  Returns the allocations that the batch holds."""
    from paper_2408_16847_gb300 import tpcf, _capi
    live = _capi.lib().tpcf_test_live_allocations
    plans, D, W, Z, N, C, G, host = [], [], [], [], [], [], [], []
    for i, (nside, k, m) in enumerate(sizes):
        edges = np.geomspace(0.2 * reach, reach, k + 1) * 58.6 / nside  # in pixels
        g = synth.rng(1300 + i)
        d = (g.standard_normal(12 * nside * nside) + 0.3).astype(np.float32)
        w = g.uniform(0.5, 1.5, len(d)).astype(np.float32)
        w[: len(w) // 5] = 0.0
        cot = g.standard_normal((m + 1, k, k))
        ct = torch.zeros((m + 1, k, k, 2), dtype=torch.float64, device="cuda:0")
        ct[..., 0] = torch.from_numpy(cot).to("cuda:0")
        plans.append(tpcf.Plan.map(nside, edges, m))
        host.append((d, w, cot, edges))
        for a, v in ((D, to_dev(d)), (W, to_dev(w)), (C, ct), (Z, torch.empty_like(ct)),
                     (N, torch.empty((k, k), dtype=torch.float64, device="cuda:0")), (G, torch.empty(len(d), device="cuda:0"))):
            a.append(v)
    before = live()
    batch = tpcf.Batch(plans, D, W, Z, N, C, G)
    held = live() - before
    for _ in range(2):
        batch.launch()
    torch.cuda.synchronize()
    for i, (nside, k, m) in enumerate(sizes):
        plans[i].sync()
        d, w, cot, edges = host[i]
        xyz = oracle.pix2vec_ring(nside)
        ref = oracle.zeta(xyz, d.astype(np.float64), w.astype(np.float64), edges, m)
        assert ref["min_margin"] > 1e-12
        assert rel_err_per_m(tpcf.as_complex(Z[i]).cpu().numpy(), ref["zeta"]).max() < TOL
        np.testing.assert_allclose(N[i].cpu().numpy(), ref["D"], rtol=1e-6, atol=1e-6 * np.abs(ref["D"]).max())
        gref = oracle.gradient(xyz, d.astype(np.float64), w.astype(np.float64), edges, m, cot.astype(np.complex128))
        assert np.abs(G[i].cpu().numpy() - gref).max() < TOL * np.abs(gref).max()
    batch.close()
    return held


def test_small_batch_has_no_workspace():
    # per member its slots, then the queue's items, the small kernels' arguments and the counters
    assert _run([(8, 1, 3), (16, 16, 4), (11, 3, 0)], 5.3) == 3 + 3


def test_large_batch():
    # linear rings (Nside 64 on) and others, and 32 bins
    assert _run([(64, 5, 6), (65, 32, 1), (20, 2, 4)], 6.1) == 3 + 4
