"""FP32 heat and KS tiers with a fixed mapping of points to threads, bit for bit against the
oracle: tiles of exactly 1, 2 and 4 pairs a thread, one more than that (the next variant, or the
tiers one by one), odd- and even-sized wide last tiles, walls, remainders, every mode."""
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


def solve(S, scheme, u0, args, nsteps, **plan):
    import torch

    sol = S.Solver(scheme, S.F32, u0.shape[-1], *args, **plan)
    u = torch.from_numpy(u0).cuda()
    sol.step(u, nsteps)
    torch.cuda.synchronize()
    sol.sync_status()
    sol.close()
    return u.cpu().numpy()


MODES = [dict(), dict(persistent=1), dict(chunk=2)]


@pytest.mark.parametrize("mode", MODES)
@pytest.mark.parametrize("threads,tile", [(32, 64), (32, 72), (32, 128), (32, 136), (32, 256), (32, 264), (64, 64),
                                          (128, 1024), (96, 8)])
@pytest.mark.parametrize("extra", [0, 1, 6])
def test_ks(S, threads, tile, extra, mode):
    n = 3 * tile + (extra if extra < tile else 0)
    p = inputs.ks_problem(n=n, seed=tile + extra, dtype=np.float32)
    steps = 3 * (tile // 4) // 2 + 3  # several passes and a remainder
    got = solve(S, S.KS, p["u0"], (p["dx"], p["dt"], p["nu"]), steps, tile_w=tile, threads=threads, **mode)
    assert np.array_equal(got, oracle.ks(p["u0"], p["dx"], p["dt"], p["nu"], steps))


@pytest.mark.parametrize("mode", MODES)
@pytest.mark.parametrize("threads,tile", [(32, 60), (32, 64), (32, 124), (32, 128), (32, 256), (64, 64), (64, 508),
                                          (64, 512), (96, 4)])
@pytest.mark.parametrize("bc,extra", [(0, 0), (0, 1), (0, 2), (1, 0), (1, 3)])
def test_heat(S, threads, tile, bc, extra, mode):
    n = 3 * tile + extra
    p = inputs.heat_problem(n=n, seed=tile + extra, dtype=np.float32)
    steps = 5 * tile // 4 + 3
    got = solve(S, S.HEAT, p["u0"], (p["dx"], p["dt"], p["alpha"]), steps, bc=bc, tile_w=tile, threads=threads, **mode)
    assert np.array_equal(got, oracle.heat(p["u0"], p["dx"], p["dt"], p["alpha"], steps, bc=bc))


@pytest.mark.parametrize("threads", [32, 64, 256])
def test_cluster(S, threads):
    p = inputs.ks_problem(n=1024, seed=5, dtype=np.float32)
    got = solve(S, S.KS, p["u0"], (p["dx"], p["dt"], p["nu"]), 77, tile_w=128, threads=threads, cluster=1)
    assert np.array_equal(got, oracle.ks(p["u0"], p["dx"], p["dt"], p["nu"], 77))
