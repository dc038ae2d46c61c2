"""tpcf_forward_noalloc beside the plan's other calls, on another stream: it shares no scratch with them."""
import ctypes

import numpy as np
import pytest
import torch

import synth
from gpu_util import TOL, rel_err_per_m, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nside", [64, 200])  # forward by tiles or few blocks, and by many blocks
def test_noalloc_overlaps_forward(cuda_device, nside):
    from paper_2408_16847_gb300 import build
    build()
    from paper_2408_16847_gb300 import _capi, tpcf
    M = 6
    plan = tpcf.Plan.map(nside, np.linspace(60.0, 60.0 * 15, 9) / nside, M)
    n = plan.npoints
    g = synth.rng(1200)
    da, db = (to_dev((g.standard_normal(n) + 0.3).astype(np.float32)) for _ in range(2))
    wa, wb = (to_dev(g.uniform(0.5, 1.5, n).astype(np.float32)) for _ in range(2))
    zeta = torch.empty(plan.zeta_shape(), dtype=torch.float64, device=cuda_device)
    norm = torch.empty((plan.K, plan.K), dtype=torch.float64, device=cuda_device)

    def noalloc(stream):
        _capi.check(_capi.lib().tpcf_forward_noalloc(plan.handle, db.data_ptr(), wb.data_ptr(), 0, n, zeta.data_ptr(),
                                                     norm.data_ptr(), ctypes.c_void_p(stream.cuda_stream)), "noalloc")

    ref_a, norm_a = plan.forward(da, wa)
    ref_b, norm_b = plan.forward(db, wb)
    torch.cuda.synchronize()
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    for _ in range(5):
        with torch.cuda.stream(s1):
            za, na = plan.forward(da, wa)
        noalloc(s2)
        torch.cuda.synchronize()
        for z, w, zr, wr in ((za, na, ref_a, norm_a), (zeta, norm, ref_b, norm_b)):
            assert rel_err_per_m(tpcf.as_complex(z).cpu().numpy(), tpcf.as_complex(zr).cpu().numpy()).max() < TOL
            np.testing.assert_allclose(w.cpu().numpy(), wr.cpu().numpy(), rtol=1e-6)
    plan.close()
