"""Euler in FP64 where the two sides of a face have nearly or exactly the same wave speed, or one
side's speed is far larger: only the faster side's is computed, so the choice must be the
oracle's maximum bit for bit.  Values far from one take the general path."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    from paper_1612_02495_gb300 import build as libbuild

    libbuild.build()
    from paper_1612_02495_gb300 import swept

    return swept


def field(kind, n, seed):
    g = np.random.Generator(np.random.Philox(seed))
    x = np.arange(n) / n
    noise = {"uniform": 0.0, "near": 1e-6, "close": 1e-9, "bits": 1e-15}.get(kind, 0.3)
    rho = 1.0 + noise * g.uniform(-1, 1, n)
    p = 1.0 + noise * g.uniform(-1, 1, n)
    u = noise * g.uniform(-1, 1, n)
    if kind == "shear":
        u = np.sin(2 * np.pi * x)
    if kind == "fast":
        u = 3.0 + 0.5 * g.uniform(-1, 1, n)
    scale = 1e-25 if kind == "tiny" else 1.0
    rho, p = rho * scale, p * scale
    return np.stack([rho, rho * u, p / 0.4 + 0.5 * rho * u * u])


@pytest.mark.parametrize("kind", ["uniform", "near", "close", "bits", "shear", "fast", "tiny"])
@pytest.mark.parametrize("bc", [0, 1])
def test_speeds(S, kind, bc):
    import torch

    n, steps = 512, 40
    U0 = field(kind, n, 11)
    dx, dt = 1.0 / n, 0.05 / n
    ref = oracle.euler(U0, dx, dt, 1.4, steps, bc=bc)
    sol = S.Solver(S.EULER, S.F64, n, dx, dt, 1.4, bc=bc, tile_w=64)
    u = torch.from_numpy(U0).cuda()
    v = u.clone()
    sol.step(u, steps)
    sol.classic(v, steps)
    torch.cuda.synchronize()
    assert np.array_equal(u.cpu().numpy().reshape(3, n), ref)
    assert np.array_equal(v.cpu().numpy().reshape(3, n), ref)
    sol.close()
