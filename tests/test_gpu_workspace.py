"""The workspace of large calls: shared by the plans of a device, separate between streams, and a plan's own
inside a graph."""
import ctypes
import threading

import numpy as np
import pytest
import torch

import synth
from gpu_util import TOL, rel_err_per_m, to_dev

pytestmark = pytest.mark.gpu

NSIDE = 200  # its passes take the block kernels
EDGES = np.linspace(0.2, 3.1, 9)


@pytest.fixture(scope="module", autouse=True)
def _built(cuda_device):
    from paper_2408_16847_gb300 import build
    build()


def _field(seed):
    g = synth.rng(seed)
    n = 12 * NSIDE * NSIDE
    return to_dev((g.standard_normal(n) + 0.3).astype(np.float32)), to_dev(g.uniform(0.5, 1.5, n).astype(np.float32))


def _same(a, b):
    from paper_2408_16847_gb300 import tpcf
    z, n = a
    zr, nr = b
    assert rel_err_per_m(tpcf.as_complex(z).cpu().numpy(), tpcf.as_complex(zr).cpu().numpy()).max() < TOL
    np.testing.assert_allclose(n.cpu().numpy(), nr.cpu().numpy(), rtol=1e-6)


def _used():
    torch.cuda.synchronize()
    free, total = torch.cuda.mem_get_info()
    return total - free


def test_many_plans_share_a_workspace():
    from paper_2408_16847_gb300 import tpcf
    edges = np.linspace(0.3, 3.1, 33)
    d, w = _field(1500)
    ref = None
    start = _used()
    plans = [tpcf.Plan.map(NSIDE, edges, 16) for _ in range(24)]
    # tables, (w d, w) and slots: 152 x 148 KB of sums and a few MB
    assert _used() - start < 24 * (64 << 20)
    for p in plans:
        out = p.forward(d, w)
        ref = ref or out
        _same(out, ref)
    assert _used() - start < 24 * (64 << 20) + (3 << 30)
    for p in plans:
        p.close()


def test_first_call_in_a_graph_and_other_plans_beside_its_replay():
    from paper_2408_16847_gb300 import tpcf
    a, b = tpcf.Plan.map(NSIDE, EDGES, 6), tpcf.Plan.map(NSIDE, EDGES, 6)
    (da, wa), (db, wb) = _field(1501), _field(1502)
    ref_a, ref_b = tpcf.Plan.map(NSIDE, EDGES, 6).forward(da, wa), b.forward(db, wb)
    za, na = torch.empty_like(ref_a[0]), torch.empty_like(ref_a[1])
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        z, n = a.forward(da, wa)
        za.copy_(z)
        na.copy_(n)
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    for _ in range(4):
        za.zero_()
        torch.cuda.synchronize()
        with torch.cuda.stream(s1):
            graph.replay()
        with torch.cuda.stream(s2):
            out = b.forward(db, wb)
        torch.cuda.synchronize()
        _same((za, na), ref_a)
        _same(out, ref_b)
    del graph
    a.close()
    b.close()


def test_threads_with_their_own_streams():
    from paper_2408_16847_gb300 import tpcf
    fields = [_field(1510 + i) for i in range(3)]
    plans = [tpcf.Plan.map(NSIDE, EDGES, 6) for _ in fields]
    g = torch.ones(plans[0].zeta_shape(), dtype=torch.float64, device="cuda:0")
    refs = []
    for p, (d, w) in zip(plans, fields):
        z, n = p.forward(d, w, (3000, 60000))  # few blocks: split into parts, the adjoint in two launches
        refs.append((z, n, p.backward(d, w, n, g, (3000, 60000))))
    torch.cuda.synchronize()
    bad = []

    def work(i):
        try:
            torch.cuda.set_device(0)
            s = torch.cuda.Stream()
            (d, w), (zr, nr, gr) = fields[i], refs[i]
            for _ in range(8):
                with torch.cuda.stream(s):
                    z, n = plans[i].forward(d, w, (3000, 60000))
                    grad = plans[i].backward(d, w, nr, g, (3000, 60000))
                s.synchronize()
                _same((z, n), (zr, nr))
                assert (grad - gr).abs().max() < TOL * gr.abs().max()
        except BaseException as e:  # noqa: BLE001
            bad.append(repr(e))

    ts = [threading.Thread(target=work, args=(i,)) for i in range(3)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not bad
    for p in plans:
        p.close()


def test_no_memory_for_a_workspace():
    from paper_2408_16847_gb300 import tpcf, _capi
    L = _capi.lib()
    plan = tpcf.Plan.map(NSIDE, EDGES, 6)
    d, w = _field(1520)
    ref = plan.forward(d, w)
    z, n = (torch.empty_like(t) for t in ref)
    args = (plan.handle, d.data_ptr(), w.data_ptr(), 0, plan.npoints, z.data_ptr(), n.data_ptr(), None,
            ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    L.tpcf_test_fail_allocation(1)
    try:
        status = L.tpcf_forward(*args)
    finally:
        L.tpcf_test_fail_allocation(0)
    assert _capi.STATUS[status] == "TPCF_ERR_OOM"
    assert L.tpcf_forward(*args) == 0
    torch.cuda.synchronize()
    plan.sync()
    _same((z, n), ref)
    plan.close()
