"""Catalogues whose bins end at fractions of a degree: pairs a millionth of the separation inside
and outside the first and the last edge are counted exactly, from tiles with many live pivots and
with one."""
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


def edge_patch(theta_deg, inner, seed, npiv=400):
    """Unit vectors: npiv pivots in a patch a few outer edges wide, and about each of them points just
    inside and outside of the outer edge and of `inner` times it, in random directions."""
    g = synth.rng(seed)
    t = np.radians(theta_deg)
    c = g.standard_normal(3)
    c /= np.linalg.norm(c)
    a = np.cross(c, [0.3, -0.5, 0.8])
    a /= np.linalg.norm(a)
    b = np.cross(c, a)
    xy = g.uniform(-4.0, 4.0, (npiv, 2)) * t
    piv = c + xy[:, :1] * a + xy[:, 1:] * b
    piv /= np.linalg.norm(piv, axis=1)[:, None]
    out = [piv]
    for r in (1.0, inner):
        for e in (-1e-4, -1e-5, -1e-6, 1e-6):
            u = g.standard_normal((npiv, 3))
            u -= (u * piv).sum(1)[:, None] * piv
            u /= np.linalg.norm(u, axis=1)[:, None]
            s = r * t * (1.0 + e)
            out.append(np.cos(s) * piv + np.sin(s) * u)
    xyz = np.concatenate(out)
    return xyz / np.linalg.norm(xyz, axis=1)[:, None]


def _case(theta, npiv):
    xyz = edge_patch(theta, 0.9, seed=1100 + int(1000 * theta), npiv=npiv)
    g = synth.rng(1101)
    d = (g.standard_normal(len(xyz)) + 0.3).astype(np.float32)
    w = g.uniform(0.5, 1.5, len(xyz)).astype(np.float32)
    return xyz, d, w, np.array([0.9, 0.95, 1.0]) * theta


THETAS = [0.005, 0.01, 0.03, 0.1, 0.5]


@pytest.mark.parametrize("theta", THETAS)
def test_edges_of_small_bins(theta):
    from paper_2408_16847_gb300 import tpcf
    xyz, d, w, edges = _case(theta, 400)
    plan = tpcf.Plan.catalog(torch.from_numpy(xyz).to("cuda:0"), edges, 3)
    counts = plan.count_pairs(to_dev(w))
    zeta, norm = plan.forward(to_dev(d), to_dev(w))
    ref = oracle.zeta(xyz, d.astype(np.float64), w.astype(np.float64), edges, 3)
    assert ref["min_margin"] > 1e-9  # (nearer to an edge, FP64 itself may differ)
    assert int(counts[0]) == int(oracle.pair_counts(xyz, edges).sum())
    np.testing.assert_allclose(norm.cpu().numpy(), ref["D"], rtol=1e-6)
    assert rel_err_per_m(tpcf.as_complex(zeta).cpu().numpy(), ref["zeta"]).max() < TOL
    plan.close()


@pytest.mark.parametrize("theta", THETAS)
def test_edges_of_small_bins_about_one_pivot(theta):
    # the cap's centre is then the pivot itself, to fp32
    from paper_2408_16847_gb300 import tpcf
    xyz, d, w, edges = _case(theta, 120)
    plan = tpcf.Plan.catalog(torch.from_numpy(xyz).to("cuda:0"), edges, 1)
    want = oracle.pair_counts(xyz, edges, pivots=np.arange(120))
    wt = to_dev(w)
    got = [plan.count_pairs(wt, (i, i + 1))[0] for i in range(120)]
    assert [int(v) for v in got] == [int(v) for v in want]
    plan.close()


@pytest.mark.parametrize("lo,hi,k", [(0.001, 20.0, 20), (0.01, 5.0, 32), (0.002, 30.0, 3)])
def test_small_edges_in_wide_tiles(lo, hi, k):
    """Sparse points with a partner each next to an edge: a tile of 32 spans tens of degrees, so its margins at the
    small edges are wider than the table's cells."""
    from paper_2408_16847_gb300 import tpcf
    g = synth.rng(1110)
    edges = np.geomspace(lo, hi, k + 1)
    a = synth.uniform_sphere(700, g)
    u = g.standard_normal(a.shape)
    u -= (u * a).sum(1)[:, None] * a
    u /= np.linalg.norm(u, axis=1)[:, None]
    s = np.radians(edges[np.arange(700) % (k + 1)] * (1.0 + g.choice([-1e-5, -1e-6, 1e-6, 1e-5], 700)))[:, None]
    b = np.cos(s) * a + np.sin(s) * u
    xyz = np.concatenate([a, b / np.linalg.norm(b, axis=1)[:, None]])
    d = (g.standard_normal(1400) + 0.3).astype(np.float32)
    w = g.uniform(0.5, 1.5, 1400).astype(np.float32)
    plan = tpcf.Plan.catalog(torch.from_numpy(xyz).to("cuda:0"), edges, 2)
    ref = oracle.zeta(xyz, d.astype(np.float64), w.astype(np.float64), edges, 2)
    assert ref["min_margin"] > 1e-9
    assert int(plan.count_pairs(to_dev(w))[0]) == int(oracle.pair_counts(xyz, edges).sum())
    _, norm = plan.forward(to_dev(d), to_dev(w))
    np.testing.assert_allclose(norm.cpu().numpy(), ref["D"], rtol=1e-6, atol=1e-6 * np.abs(ref["D"]).max())
    plan.close()
