"""2D heat with the plan left to the library (overlapped tiles): bit for bit the oracle's values.
Grids smaller than a window, not square, with partly filled last tiles; one step, fewer and more
than a launch's steps, and runs long enough to replay the cached launches."""
import numpy as np
import pytest

import oracle
from paper_1612_02495_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    from paper_1612_02495_gb300 import build as libbuild

    libbuild.build()
    from paper_1612_02495_gb300 import swept

    return swept


@pytest.mark.parametrize("npd", [np.float32, np.float64])
@pytest.mark.parametrize("bc", [0, 1])
@pytest.mark.parametrize("nx,ny,calls", [(16, 16, (1, 2, 40)), (24, 200, (3, 61)), (96, 40, (5, 8)), (256, 64, (7, 1)),
                                         (520, 376, (33,)), (768, 512, (12,)), (64, 64, (1500,)), (1024, 1056, (9,))])
def test_parity(S, nx, ny, calls, bc, npd):
    import torch

    p = inputs.heat2d_problem(nx=nx, ny=ny, seed=nx + ny, dtype=npd)
    sol = S.Solver2D(S.F32 if npd == np.float32 else S.F64, nx, ny, p["dx"], p["dt"], p["alpha"], bc=bc)
    u = torch.from_numpy(p["u0"]).cuda()
    for n in calls:
        sol.step(u, n)
    torch.cuda.synchronize()
    sol.sync_status()
    sol.close()
    ref = oracle.heat2d(p["u0"], p["dx"], p["dt"], p["alpha"], sum(calls), bc=bc, threads=8)
    assert np.array_equal(u.cpu().numpy(), ref)


@pytest.mark.parametrize("npd", [np.float32, np.float64])
@pytest.mark.parametrize("zero", ["all", "half", "points", "wide"])
def test_zeros_and_range(S, zero, npd):
    """fields with zeros, signed zeros, subnormals and a wide range of magnitudes"""
    import torch

    g = np.random.Generator(np.random.Philox(7))
    u0 = g.uniform(-1, 1, (96, 128)).astype(npd)
    if zero == "all":
        u0[:] = 0
    elif zero == "half":
        u0[:, 50:] = 0
        u0[40:60, 90:] = -0.0
    elif zero == "points":
        u0[::7, ::5] = 0
    else:
        u0 *= (10.0 ** g.uniform(-300 if npd == np.float64 else -44, 0, u0.shape)).astype(npd)
    sol = S.Solver2D(S.F32 if npd == np.float32 else S.F64, 128, 96, 1.0, 0.2, 1.0)
    u = torch.from_numpy(u0).cuda()
    sol.step(u, 21)
    torch.cuda.synchronize()
    sol.close()
    assert np.array_equal(u.cpu().numpy(), oracle.heat2d(u0, 1.0, 0.2, 1.0, 21))
