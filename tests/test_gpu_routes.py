"""Both sets of map kernels (tiles for calls with little work, blocks for the others) on every form of
call, against the FP64 oracle, and the choice between them.

Nside 64: its belt rings have the 256 pixels that a linear block holds, the outer edge of 6 degrees leaves
rings of both classes, and the pivot range cuts rings, blocks and tiles of both."""
import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_util import TOL, rel_err_per_m, to_dev
from test_gpu_blocks import _check_step

pytestmark = pytest.mark.gpu

TILES, BLOCKS = 1, 2
NSIDE, M = 64, 5
CAP = 2 * NSIDE * (NSIDE - 1)
EDGES = np.geomspace(1.03, 5.9, 7)
# the cap's last rings and the belt's first; the belt's middle across pixel 0 of rings; few pivots of a ring
RANGES = [(CAP - 700, CAP + 1500), (CAP + 16384 - 300, CAP + 16384 + 500), (CAP + 20000, CAP + 20033)]


@pytest.fixture(scope="module", autouse=True)
def _built(cuda_device):
    from paper_2408_16847_gb300 import build
    build()


def plan_on(route, *a, **k):
    from paper_2408_16847_gb300 import tpcf, _capi
    p = tpcf.Plan.map(*a, **k)
    assert _capi.lib().tpcf_test_route(p.handle, route) == 0
    return p


@pytest.fixture(scope="module")
def field():
    d = synth.bump_map(NSIDE, 300, (1.0, 6.0), 0.5, 0.05, seed=synth.BASE_SEED + 90).astype(np.float32)
    w = synth.rng(91).uniform(0.5, 1.5, len(d)).astype(np.float32)
    return oracle.pix2vec_ring(NSIDE), d, w


def _zeta(t):
    from paper_2408_16847_gb300 import tpcf
    return tpcf.as_complex(t).cpu().numpy()


@pytest.mark.parametrize("route", [TILES, BLOCKS])
@pytest.mark.parametrize("pivots", RANGES)
def test_forward_and_adjoint(route, pivots, field):
    xyz, d, w = field
    plan = plan_on(route, NSIDE, EDGES, M)
    _check_step(plan, xyz, d, w, EDGES, M, pivots)
    plan.close()


@pytest.mark.parametrize("route", [TILES, BLOCKS])
@pytest.mark.parametrize("pivots", RANGES)
def test_self_pair_subtraction(route, pivots, field):
    xyz, d, w = field
    K, piv = len(EDGES) - 1, np.arange(*pivots)
    plan = plan_on(route, NSIDE, EDGES, M, self_pairs="subtract")
    dd, ww = d.astype(np.float64), w.astype(np.float64)
    ref = oracle.zeta(xyz, dd, ww, EDGES, M, pivots=piv, self_pairs="subtract")
    dt, wt = to_dev(d), to_dev(w)
    zeta, norm = plan.forward(dt, wt, pivots)
    assert rel_err_per_m(_zeta(zeta), ref["zeta"]).max() < TOL
    np.testing.assert_allclose(norm.cpu().numpy(), ref["D"], rtol=1e-6, atol=1e-6 * np.abs(ref["D"]).max())
    cot = synth.rng(92).standard_normal((M + 1, K, K))
    g = torch.zeros((M + 1, K, K, 2), dtype=torch.float64, device=dt.device)
    g[..., 0] = torch.from_numpy(cot).to(dt.device)
    grad = plan.backward(dt, wt, norm, g, pivots)
    plan.sync()
    gref = oracle.gradient(xyz, dd, ww, EDGES, M, cot.astype(np.complex128), pivots=piv, self_pairs="subtract")
    assert np.abs(grad.cpu().numpy() - gref).max() < TOL * np.abs(gref).max()
    plan.close()


@pytest.mark.parametrize("route", [TILES, BLOCKS])
@pytest.mark.parametrize("norm,reading", [("bin_mean", "R2"), ("pivot_total", "R1")])
def test_pivot_normalisation(route, norm, reading, field):
    xyz, d, w = field
    plan = plan_on(route, NSIDE, EDGES, M, norm=norm)
    for pivots in RANGES:
        ref = oracle.zeta(xyz, d.astype(np.float64), w.astype(np.float64), EDGES, M, pivots=np.arange(*pivots), norm=reading)
        zeta, _ = plan.forward(to_dev(d), to_dev(w), pivots)
        assert rel_err_per_m(_zeta(zeta), ref["zeta"]).max() < TOL
    plan.close()


@pytest.mark.parametrize("route", [TILES, BLOCKS])
def test_tensor_core_contraction(route, field):
    xyz, d, w = field
    plan = plan_on(route, NSIDE, EDGES, M, contract="tc")
    for pivots in RANGES:
        ref = oracle.zeta(xyz, d.astype(np.float64), w.astype(np.float64), EDGES, M, pivots=np.arange(*pivots))
        zeta, _ = plan.forward(to_dev(d), to_dev(w), pivots)
        plan.sync()
        assert rel_err_per_m(_zeta(zeta), ref["zeta"]).max() < TOL
    plan.close()


@pytest.mark.parametrize("route", [TILES, BLOCKS])
@pytest.mark.parametrize("group", [2, 15])
def test_shared_neighbour_lists(route, group, field):
    xyz, d, w = field
    plan = plan_on(route, NSIDE, EDGES, M)
    for pivots in RANGES + [(0, len(d))]:
        ref = oracle.zeta_grouped(NSIDE, d.astype(np.float64), w.astype(np.float64), EDGES, M, group, pivots=np.arange(*pivots))
        zeta, norm = plan.forward_grouped(to_dev(d), to_dev(w), group, pivots)
        assert rel_err_per_m(_zeta(zeta), ref["zeta"]).max() < TOL
        np.testing.assert_allclose(norm.cpu().numpy(), ref["D"], rtol=1e-6, atol=1e-6 * np.abs(ref["D"]).max())
    plan.close()


@pytest.mark.parametrize("route", [TILES, BLOCKS])
def test_three_fields(route, field):
    xyz, _, _ = field
    fields = []
    for f in range(3):
        g = synth.rng(93 + f)
        fields.append(((g.standard_normal(len(xyz)) + 0.3).astype(np.float32),
                       g.uniform(0.5, 1.5, len(xyz)).astype(np.float32)))
    plan = plan_on(route, NSIDE, EDGES, M)
    for pivots in RANGES:
        zeta, norm = plan.forward_multi([(to_dev(d), to_dev(w)) for d, w in fields], pivots)
        ref = oracle.zeta_multi(xyz, [(d.astype(np.float64), w.astype(np.float64)) for d, w in fields], EDGES, M,
                                pivots=np.arange(*pivots))
        assert rel_err_per_m(_zeta(zeta), ref["zeta"]).max() < TOL
        np.testing.assert_allclose(norm.cpu().numpy(), ref["D"], rtol=1e-6, atol=1e-6 * np.abs(ref["D"]).max())
    plan.close()


@pytest.mark.parametrize("nside", [63, 65])
@pytest.mark.parametrize("k,m", [(1, 0), (32, 3), (3, 16)])
def test_block_edges(nside, k, m):
    # rings one pixel group short of and past a linear block, the smallest and largest bins and multipoles
    d = synth.bump_map(nside, 200, (1.0, 6.0), 0.5, 0.05, seed=synth.BASE_SEED + 40).astype(np.float32)
    w = synth.rng(41).uniform(0.5, 1.5, len(d)).astype(np.float32)
    edges = np.geomspace(1.03, 5.9, k + 1)
    xyz = oracle.pix2vec_ring(nside)
    plan = plan_on(BLOCKS, nside, edges, m)
    belt = 2 * nside * (nside - 1) + 4 * nside * nside
    for lo, n in ((belt - 37, 300), (belt + 255, 2), (2 * nside * (nside - 1) - 150, 301), (0, 90)):
        _check_step(plan, xyz, d, w, edges, m, (lo, lo + n))
    plan.close()


def _launches(plan, call):
    before = plan.kernel_launches()
    call()
    return plan.kernel_launches() - before


def test_small_calls_are_not_split():
    """A call with little work goes to the tile kernels: its adjoint is the preparation and one kernel (the
    blocks' takes two, one for each half of its phases)."""
    from paper_2408_16847_gb300 import tpcf
    plan = tpcf.Plan.map(16, [1.3, 12.1], 4)
    d = to_dev(synth.rng(94).standard_normal(12 * 16 * 16).astype(np.float32))
    w = torch.ones_like(d)
    _, norm = plan.forward(d, w)
    g = torch.ones(plan.zeta_shape(), dtype=torch.float64, device=d.device)
    assert _launches(plan, lambda: plan.backward(d, w, norm, g)) == 2
    plan.close()
    plan = tpcf.Plan.map(24, np.linspace(1.3, 24.0, 5), 4)
    d = to_dev(synth.rng(95).standard_normal(12 * 24 * 24).astype(np.float32))
    w = torch.ones_like(d)
    _, norm = plan.forward(d, w)
    g = torch.ones(plan.zeta_shape(), dtype=torch.float64, device=d.device)
    assert _launches(plan, lambda: plan.backward(d, w, norm, g)) == 2
    plan.close()


@pytest.mark.parametrize("bins", [2, 9])
def test_small_contributions_reach_the_fp64_sums(bins):
    """At most 64 pivots of a linear block are added up in fp32: 64 pivots of weight 2^-30 beside 64 of weight 1
    keep their share of D, which sums in fp32 over 128 pivots lose."""
    n = 12 * NSIDE * NSIDE
    first = CAP + 4 * NSIDE * NSIDE  # pixel 0 of the equator: the block's first
    w = np.ones(n, dtype=np.float32)
    w[first + 64:first + 128] = 2.0 ** -30
    d, w = to_dev(np.ones(n, dtype=np.float32)), to_dev(w)
    plan = plan_on(BLOCKS, NSIDE, np.linspace(1.03, 5.9, bins + 1), 1)
    whole, large, small = (plan.forward(d, w, (first + a, first + b))[1].cpu().numpy() for a, b in ((0, 128), (0, 64), (64, 128)))
    plan.sync()
    np.testing.assert_allclose(whole - large, small, rtol=1e-6)
    plan.close()


def test_linear_rings_of_several_blocks():
    """Nside 256: four blocks to a ring, in the ring's middle (no row wraps) and across pixel 0."""
    nside, m = 256, 6
    edges = np.geomspace(0.31, 1.47, 6)
    d = synth.bump_map(nside, 2000, (0.3, 2.0), 0.5, 0.05, seed=synth.BASE_SEED + 96).astype(np.float32)
    w = synth.rng(97).uniform(0.5, 1.5, len(d)).astype(np.float32)
    xyz = oracle.pix2vec_ring(nside)
    plan = plan_on(BLOCKS, nside, edges, m)
    ring = 2 * nside * (nside - 1) + 4 * nside * nside
    for pivots in ((ring + 400, ring + 640), (ring + 511, ring + 514), (ring - 60, ring + 40)):
        _check_step(plan, xyz, d, w, edges, m, pivots)
    plan.close()


def _exact_sums(nside, edges, m, field, pivots, cot):
    """zeta, D and the gradient in 64 bits, from the workload file's direct sums over the pivots' rings."""
    import importlib.util
    import os
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    spec = importlib.util.spec_from_file_location("cases", os.path.join(root, "perf", "cases.py"))
    cases = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(cases)
    cases.edges_of = lambda case: np.array(edges)
    case = dict(kind="map_host", k=len(edges) - 1, m=m, opt="default")
    return cases.exact_sums(case, cases.Map(nside, np.radians(edges[-1])), [field], pivots, cot)


# a warp's gradient rows fit its shared memory (reach 989 pixels), or go straight to the gradient (1018, 1054)
@pytest.mark.parametrize("outer", [20.9, 21.5, 22.2])
def test_wide_gradient_rows(outer):
    nside, m = 4096, 3
    edges = [outer - 0.1, outer - 0.04, outer]
    n = 12 * nside * nside
    first = 2 * nside * (nside - 1) + 4 * nside * nside + 5000
    pivots = (first, first + 300)
    g = torch.Generator(device="cuda:0")
    g.manual_seed(98)
    d = torch.randn(n, generator=g, device="cuda:0") + 0.3
    w = 0.5 + torch.rand(n, generator=g, device="cuda:0")
    cot = torch.randn(m + 1, 2, 2, 2, generator=g, device="cuda:0", dtype=torch.float64)
    cot[..., 1] = 0.0
    plan = plan_on(BLOCKS, nside, edges, m)
    zeta, norm = plan.forward(d, w, pivots)
    grad = plan.backward(d, w, norm, cot, pivots)
    plan.sync()
    plan.close()
    ref = _exact_sums(nside, edges, m, (d, w), pivots, cot)
    zref = torch.view_as_complex(ref["zeta"].contiguous()).cpu().numpy()
    assert rel_err_per_m(_zeta(zeta), zref).max() < TOL
    np.testing.assert_allclose(norm.cpu().numpy(), ref["norm"].cpu().numpy(), rtol=1e-6)
    assert (grad.double() - ref["grad"]).abs().max() < TOL * ref["grad"].abs().max()
