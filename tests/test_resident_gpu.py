"""Small heat and KS grids with the plan left to the library (the resident kernel): equal bit
for bit to the oracle.  Sizes: the smallest tiled grid, fewer points than lanes, odd sizes with
a partly filled last warp, one block and clusters of up to 16, both sides of the rule's limits.
Steps: one, fewer and more than a trade interval, odd counts."""
import os

import numpy as np
import pytest

import oracle
from paper_1612_02495_gb300 import inputs

pytestmark = pytest.mark.gpu

THREADS = max(1, min(32, os.cpu_count() or 1))
HEAT_N = (8, 17, 33, 100, 1009, 1024, 4096, 5001, 32768, 40001)
KS_N = (16, 33, 100, 1009, 2048, 4097, 16384, 24001)


@pytest.fixture(scope="module")
def S():
    from paper_1612_02495_gb300 import build as libbuild

    libbuild.build()
    from paper_1612_02495_gb300 import swept

    return swept


def solve(S, scheme, dtype, u0, args, bc, steps):
    import torch

    sol = S.Solver(scheme, dtype, u0.shape[-1], *args, bc=bc)
    u = torch.from_numpy(u0).cuda()
    for n in steps:
        sol.step(u, n)
    torch.cuda.synchronize()
    sol.sync_status()
    sol.close()
    return u.cpu().numpy()


@pytest.mark.parametrize("npd", [np.float32, np.float64])
@pytest.mark.parametrize("bc", [0, 1])
@pytest.mark.parametrize("n", HEAT_N)
def test_heat(S, n, bc, npd):
    p = inputs.heat_problem(n=n, seed=n, dtype=npd)
    dtype = S.F32 if npd == np.float32 else S.F64
    got = solve(S, S.HEAT, dtype, p["u0"], (p["dx"], p["dt"], p["alpha"]), bc, (1, 2, 131))
    ref = oracle.heat(p["u0"], p["dx"], p["dt"], p["alpha"], 134, bc=bc)
    assert np.array_equal(got, ref)


@pytest.mark.parametrize("npd", [np.float32, np.float64])
@pytest.mark.parametrize("n", KS_N)
def test_ks(S, n, npd):
    p = inputs.ks_problem(n=n, seed=n, dtype=npd)
    dtype = S.F32 if npd == np.float32 else S.F64
    got = solve(S, S.KS, dtype, p["u0"], (p["dx"], p["dt"], p["nu"]), 0, (1, 2, 67))
    assert np.array_equal(got, oracle.ks(p["u0"], p["dx"], p["dt"], p["nu"], 70, threads=THREADS))


def test_captured(S):
    """the call is one launch on the caller's stream, also into a capture"""
    import torch

    p = inputs.heat_problem(n=1009, seed=3)
    sol = S.Solver(S.HEAT, S.F64, 1009, p["dx"], p["dt"], p["alpha"])
    u0 = torch.from_numpy(p["u0"]).cuda()
    u = u0.clone()
    sol.step(u, 5)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        u.copy_(u0)
        sol.step(u, 77)
    for _ in range(2):
        g.replay()
    torch.cuda.synchronize()
    assert np.array_equal(u.cpu().numpy(), oracle.heat(p["u0"], p["dx"], p["dt"], p["alpha"], 77))
    sol.close()
