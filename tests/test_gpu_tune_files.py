"""Stored launch configurations: what the tile kernels' keys (v2) name is read as it was written, and the
register variants and CTA counts that fit are those of the kernels."""
import numpy as np
import pytest
import torch

import synth
from gpu_util import to_dev

pytestmark = pytest.mark.gpu


def _tpcf():
    from paper_2408_16847_gb300 import build
    build()
    from paper_2408_16847_gb300 import tpcf
    return tpcf


def _field(nside):
    d = to_dev(synth.rng(1400).standard_normal(12 * nside * nside).astype(np.float32))
    return d, torch.ones_like(d)


@pytest.mark.parametrize("nside,key", [(16, "v2 "), (200, "v4 ")])  # tiles; blocks
def test_key_names_the_kernels(cuda_device, tmp_path, monkeypatch, nside, key):
    tpcf = _tpcf()
    cache = tmp_path / "tune.txt"
    monkeypatch.setenv("TPCF_AUTOTUNE_CACHE", str(cache))
    edges = np.linspace(30.0, 300.0, 9) / nside
    plan = tpcf.Plan.map(nside, edges, 3)
    plan.autotune(*_field(nside))
    line = cache.read_text()
    assert line.startswith(key)
    # another configuration under the same key, as a program may have stored it
    cache.write_text(line.split("|")[0] + "| fwd 2 1 4 1 bwd 3 1 16\n")
    again = tpcf.Plan.map(nside, edges, 3)
    assert again.launch_config() == {"forward": {"variant": 2, "ctas_per_sm": 1, "flush_rings": 4, "quarter_turn_tiles": 1},
                                     "adjoint": {"variant": 3, "ctas_per_sm": 1, "flush_rings": 16}}
    for p in (plan, again):
        p.close()


def test_configurations_that_do_not_fit_are_refused(cuda_device):
    # one tile of 32 bins and 16 multipoles fills an SM's shared memory
    tpcf = _tpcf()
    plan = tpcf.Plan.map(16, np.linspace(1.3, 20.0, 33), 16)
    base = plan.launch_config()
    assert base["forward"]["ctas_per_sm"] == base["adjoint"]["ctas_per_sm"] == 1
    one = {"variant": 3, "ctas_per_sm": 2, "flush_rings": 8}
    with pytest.raises(Exception) as e:
        plan.set_launch_config({"forward": dict(one, quarter_turn_tiles=0), "adjoint": one})
    assert getattr(e.value, "status", None) == 1
    assert plan.launch_config() == base
    plan.close()
