"""What a recorded launch plan is good for (aim_opts.autotune, the plan cache).

* A plan recorded under the key of other kernels (no path of the grid passes, no box, no
  revision in it) is not taken for this library's: the set-up measures its own.
* A plan of the same transform lengths but another box is another plan.
* Fields that the context's kernels have no choice in (k_zwarp, k_ypipe) keep the defaults
  instead of recording the noise of timing one kernel several times.
"""
import json

import numpy as np
import pytest

from paper_1408_7060_gb300.inputs import icosphere, make_workload, place_grid

pytestmark = pytest.mark.gpu

FIELDS = ("zw", "cw", "rp", "ypb")


def test_a_plan_of_other_kernels_is_measured_anew(tmp_path, monkeypatch):
    import torch

    from paper_1408_7060_gb300 import AimContext, abi

    cache = tmp_path / "plans.jsonl"
    monkeypatch.setenv("AIM_GB300_PLAN_CACHE", str(cache))
    name = torch.cuda.get_device_name().replace('"', "_").replace("|", "_")
    w = make_workload("sphere_sub3_n32")
    with AimContext.from_workload(w) as c:
        lz = c.info["z_len"]
    cache.write_text(json.dumps({"key": f"{name}|L=64|LZ={lz}|prec=c64|nb={w.nb}", "zw": 16, "cw": 16, "rp": 64,
                                 "ypb": 8}) + "\n")
    with AimContext.from_workload(w, autotune=1) as c:
        assert c.info["plan_source"] == abi.AIM_PLAN_MEASURED
    key = json.loads(cache.read_text().splitlines()[-1])["key"]
    assert key.startswith(name) and "|path=plane|" in key
    with AimContext.from_workload(w, autotune=1) as c:
        assert c.info["plan_source"] == abi.AIM_PLAN_CACHED


def flat(z, batch_max=1, **kw):
    from paper_1408_7060_gb300 import AimContext

    V, F = icosphere(2, 1.0)
    V = V * np.array([1.0, 1.0, z])
    h, origin = place_grid(V, 128)
    return AimContext(V=V, F=F, grid_n=128, origin=origin, h=h, near_radius=3 * h, dt=0.25 / 90e6, f_c=300e6,
                      precision="c64", batch_max=batch_max, **kw)


def test_fields_without_a_choice_keep_the_defaults(tmp_path, monkeypatch):
    from paper_1408_7060_gb300 import abi

    monkeypatch.setenv("AIM_GB300_PLAN_CACHE", str(tmp_path / "plans.jsonl"))
    with flat(0.7) as c:
        assert c.info["z_len"] == 192
        plan, nz = {k: c.info["plan_" + k] for k in FIELDS}, c.info["box_hi"][2] - c.info["box_lo"][2]
    with flat(0.7, autotune=2) as c:
        assert c.info["plan_source"] == abi.AIM_PLAN_MEASURED
        assert all(c.info["plan_" + k] == plan[k] for k in ("zw", "cw"))
    with flat(0.65, autotune=1) as c:                       # the same lengths, fewer box planes
        assert c.info["z_len"] == 192 and c.info["box_hi"][2] - c.info["box_lo"][2] < nz
        assert c.info["plan_source"] == abi.AIM_PLAN_MEASURED
