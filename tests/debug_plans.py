"""Solves with the plan left to the library under the debug build (SWEPT_DEBUG=1), called by
test_debug_plans.py in a child process: the resident kernel (one block and a cluster, both walls,
partly filled last warps) and 2D overlapped tiles (partly filled last tiles, zeros), FP64 KS tiers on
fields that go over to FP64.  The device-side index checks must stay clean and every result
must equal the oracle bit for bit."""
import os
import sys

import numpy as np

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import oracle  # noqa: E402
from paper_1612_02495_gb300 import inputs  # noqa: E402


def main():
    import torch

    from paper_1612_02495_gb300 import swept as S

    assert S.DEBUG_BUILD

    def run(sol, u0, nsteps, ref, what):
        u = torch.from_numpy(np.ascontiguousarray(u0)).cuda()
        sol.step(u, nsteps)
        torch.cuda.synchronize()
        _, rec = S.debug_status()
        assert rec is None, (what, rec)
        assert np.array_equal(u.cpu().numpy(), ref), what
        sol.close()
        print("clean:", what, flush=True)

    for npd, code in ((np.float64, S.F64), (np.float32, S.F32)):
        for n, bc in ((8, 0), (33, 1), (1009, 1), (4096, 0)):
            p = inputs.heat_problem(n=n, dtype=npd)
            ref = oracle.heat(p["u0"], p["dx"], p["dt"], p["alpha"], 131, bc=bc)
            run(S.Solver(S.HEAT, code, n, p["dx"], p["dt"], p["alpha"], bc=bc), p["u0"], 131, ref, ("heat", n, bc, code))
        for n in (16, 1009, 2048):
            p = inputs.ks_problem(n=n, dtype=npd)
            ref = oracle.ks(p["u0"], p["dx"], p["dt"], p["nu"], 67)
            run(S.Solver(S.KS, code, n, p["dx"], p["dt"], p["nu"]), p["u0"], 67, ref, ("ks", n, code))
        for nx, ny, bc in ((16, 16, 0), (96, 40, 1), (512, 144, 0)):
            p = inputs.heat2d_problem(nx=nx, ny=ny, dtype=npd)
            u0 = np.where(np.arange(nx) % 9 < 4, p["u0"], 0).astype(npd)
            ref = oracle.heat2d(u0, p["dx"], p["dt"], p["alpha"], 23, bc=bc, threads=8)
            run(S.Solver2D(code, nx, ny, p["dx"], p["dt"], p["alpha"], bc=bc), u0, 23, ref, ("heat2d", nx, ny, bc, code))
    for kw in (dict(tile_w=64), dict(tile_w=32, threads=64, persistent=1), dict(tile_w=128, threads=32)):
        p = inputs.ks_problem(n=1027)
        u0 = np.where(np.arange(1027) < 700, 0.5, p["u0"])
        ref = oracle.ks(u0, p["dx"], p["dt"], p["nu"], 67)
        run(S.Solver(S.KS, S.F64, 1027, p["dx"], p["dt"], p["nu"], **kw), u0, 67, ref, ("ks fields", kw))
    print("all clean")


if __name__ == "__main__":
    main()
