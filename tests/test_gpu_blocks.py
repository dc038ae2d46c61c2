"""The pair kernels' work splits at the sizes where they change: rings about the length of a
block of 256 pivots, pivot ranges that cut blocks and rings, the smallest and largest numbers of
bins and multipoles, catalogues about a batch of candidates; against the FP64 oracle.

The bar is the library's stated accuracy, TOL per multipole (fp32 moments: a sum of n terms in
runs of at most 256 carries about 256 x 6e-8 = 1.5e-5 of a single term's size at worst and
sqrt(256) x 6e-8 = 1e-6 typically)."""
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


def _tpcf():
    from paper_2408_16847_gb300 import tpcf
    return tpcf


def _check_step(plan, xyz, d, w, edges, M, pivots):
    """zeta, D and the gradient over a pivot range against the oracle."""
    tpcf = _tpcf()
    K = len(edges) - 1
    piv = np.arange(*pivots)
    ref = oracle.zeta(xyz, d.astype(np.float64), w.astype(np.float64), edges, M, pivots=piv)
    assert ref["min_margin"] > 1e-12
    dt, wt = to_dev(d), to_dev(w)
    zeta, norm = plan.forward(dt, wt, pivots)
    cot = synth.rng(31).standard_normal((M + 1, K, K))
    g = torch.zeros((M + 1, K, K, 2), dtype=torch.float64, device=dt.device)
    g[..., 0] = torch.from_numpy(cot).to(dt.device)
    grad = plan.backward(dt, wt, norm, g, pivots)
    plan.sync()
    e = rel_err_per_m(tpcf.as_complex(zeta).cpu().numpy(), ref["zeta"])
    assert e.max() < TOL, "zeta %s" % np.array2string(e, precision=2)
    np.testing.assert_allclose(norm.cpu().numpy(), ref["D"], rtol=1e-6, atol=1e-6 * np.abs(ref["D"]).max())
    gref = oracle.gradient(xyz, d.astype(np.float64), w.astype(np.float64), edges, M, cot.astype(np.complex128),
                           pivots=piv)
    assert np.abs(grad.cpu().numpy() - gref).max() < TOL * np.abs(gref).max()


@pytest.mark.parametrize("nside", [63, 64, 65])  # belt rings of 252, 256 and 260 pixels
@pytest.mark.parametrize("k,M", [(1, 0), (5, 7), (32, 3)])
def test_block_edges_on_maps(nside, k, M):
    d = synth.bump_map(nside, 200, (1.0, 6.0), 0.5, 0.05, seed=synth.BASE_SEED + 40).astype(np.float32)
    w = synth.rng(41).uniform(0.5, 1.5, len(d)).astype(np.float32)
    edges = np.geomspace(1.03, 5.9, k + 1)
    xyz = oracle.pix2vec_ring(nside)
    plan = _tpcf().Plan.map(nside, edges, M)
    belt = 2 * nside * (nside - 1) + 4 * nside * nside  # first pixel of the equator
    for lo, n in ((belt - 37, 300), (belt + 255, 2), (2 * nside * (nside - 1) - 150, 301), (0, 90)):
        _check_step(plan, xyz, d, w, edges, M, (lo, lo + n))
    plan.close()


@pytest.mark.parametrize("n", [1, 31, 33, 511, 513, 1025])
@pytest.mark.parametrize("k,M", [(1, 16), (9, 2), (32, 5)])
def test_batch_edges_on_catalogues(n, k, M):
    # all points within 2 degrees: every tile has every point as a candidate
    g = synth.rng(50 + n)
    a, b = g.uniform(-0.017, 0.017, (2, n))
    xyz = np.stack([np.cos(b) * np.cos(a), np.cos(b) * np.sin(a), np.sin(b)], 1)
    d = (g.standard_normal(n) + 0.3).astype(np.float32)
    w = g.uniform(0.5, 1.5, n).astype(np.float32)
    edges = np.linspace(0.2, 4.1, k + 1)
    plan = _tpcf().Plan.catalog(torch.from_numpy(xyz).to("cuda:0"), edges, M)
    if n == 1:  # no pair at all
        zeta, norm = plan.forward(to_dev(d), to_dev(w))
        assert torch.all(zeta == 0) and torch.all(norm == 0)
    else:
        _check_step(plan, xyz, d, w, edges, M, (0, n))
    plan.close()


def test_three_ctas_configuration_is_accepted():
    tpcf = _tpcf()
    plan = tpcf.Plan.map(16, [1.3, 4.1, 9.7], 3)
    one = {"variant": 3, "ctas_per_sm": 3, "flush_rings": 8}
    cfg = {"forward": dict(one, quarter_turn_tiles=0), "adjoint": one}
    base = plan.launch_config()
    d = to_dev(synth.rng(60).standard_normal(12 * 16 * 16).astype(np.float32))
    w = torch.ones_like(d)
    z0, _ = plan.forward(d, w)
    z0 = z0.clone()
    plan.set_launch_config(cfg)
    assert plan.launch_config() == cfg
    z1, _ = plan.forward(d, w)
    plan.sync()
    assert (z1 - z0).abs().max() < TOL * z0.abs().max()
    plan.set_launch_config(base)
    plan.close()


@pytest.mark.parametrize("kind", ["map", "catalog"])
@pytest.mark.parametrize("k,M", [(31, 1), (32, 0), (32, 6)])
def test_three_fields_at_the_most_bins(kind, k, M):
    # the contraction's stage is full at 32 bins
    tpcf = _tpcf()
    edges = np.geomspace(2.03, 17.9, k + 1)
    if kind == "map":
        xyz = oracle.pix2vec_ring(32)
        plan = tpcf.Plan.map(32, edges, M)
    else:
        xyz = synth.uniform_sphere(3000, synth.rng(70))
        plan = tpcf.Plan.catalog(torch.from_numpy(xyz).to("cuda:0"), edges, M)
    fields = []
    for f in range(3):
        g = synth.rng(71 + f)
        fields.append(((g.standard_normal(len(xyz)) + 0.3).astype(np.float32),
                       g.uniform(0.5, 1.5, len(xyz)).astype(np.float32)))
    pivots = (0, len(xyz)) if kind == "catalog" else (4000, 6500)
    zeta, norm = plan.forward_multi([(to_dev(d), to_dev(w)) for d, w in fields], pivots)
    plan.sync()
    ref = oracle.zeta_multi(xyz, [(d.astype(np.float64), w.astype(np.float64)) for d, w in fields], edges, M,
                            pivots=np.arange(*pivots))
    assert ref["min_margin"] > 1e-12
    assert rel_err_per_m(tpcf.as_complex(zeta).cpu().numpy(), ref["zeta"]).max() < TOL
    np.testing.assert_allclose(norm.cpu().numpy(), ref["D"], rtol=1e-6, atol=1e-6 * np.abs(ref["D"]).max())
    plan.close()
