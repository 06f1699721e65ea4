"""The tuner's plan is never slower than leaving the plan to the library, which has kernels of its
own for small 1D grids and for 2D, and a cache written for older kernels is not used."""
import json

import numpy as np
import pytest

from paper_1612_02495_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mods():
    from paper_1612_02495_gb300 import build as libbuild

    libbuild.build()
    from paper_1612_02495_gb300 import autotune
    from paper_1612_02495_gb300 import swept as S

    return S, autotune


@pytest.mark.parametrize("f64", [False, True])
def test_small_heat(mods, f64, tmp_path):
    import torch

    S, autotune = mods
    code = S.F64 if f64 else S.F32
    cache = tmp_path / "tune.json"
    old = {"single4/%s/%d/%d/%d/%s/%d" % (autotune._device_key(), S.HEAT, code, 1024, 2000, 1): {"tile_w": 4, "threads": 32}}
    cache.write_text(json.dumps(old))
    plan = autotune.tune_single(S.HEAT, code, 1024, probe_steps=2000, cache=str(cache))
    assert plan["tile_w"] == 0 and plan["threads"] == 0  # the resident kernel: 2 to 4 times any explicit plan
    assert autotune.tune_single(S.HEAT, code, 1024, probe_steps=2000, cache=str(cache)) == plan
    p = inputs.heat_problem(n=1024, dtype=np.float64 if f64 else np.float32)
    sol = autotune.solver_from_plan(S.HEAT, code, 1024, p["dx"], p["dt"], p["alpha"], plan)
    u = torch.from_numpy(p["u0"]).cuda()
    v = u.clone()
    sol.step(u, 500)
    sol.classic(v, 500)
    torch.cuda.synchronize()
    assert torch.equal(u, v)
    sol.close()


def test_2d(mods):
    S, autotune = mods
    plan = autotune.tune_2d(S.F32, 512, 512, cache=None)
    assert plan["tile_w"] == 0 and plan["persistent"] == 0  # overlapped tiles: 2 to 4 times any swept plan
