"""A batch in blocks of 64 threads costs no more than twice one of 256: with four pairs of points a
lane inlined into the batch kernel it took 2.5 to 3 times as long."""
import numpy as np
import pytest

from paper_1612_02495_gb300 import inputs

pytestmark = pytest.mark.gpu


def test_threads():
    import torch

    from paper_1612_02495_gb300 import build as libbuild

    libbuild.build()
    from paper_1612_02495_gb300 import swept as S

    spec = inputs.batch_problems(count=66, seed=66, log2_hi=14, steps_lo=60, steps_hi=300)
    probs, ms = inputs.batch_instances(spec, dtype=np.float32), {}
    for threads in (64, 256):
        b = S.Batch(probs, S.F32, threads=threads)
        u0 = b.pack([q["u0"] for q in probs])
        u = u0.clone()
        for _ in range(4):  # the first one warms up
            u.copy_(u0)
            a, e = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            b.run(u)
            e.record()
            torch.cuda.synchronize()
            ms.setdefault(threads, []).append(a.elapsed_time(e))
        b.close()
    assert min(ms[64][1:]) < 2 * min(ms[256][1:]), ms
