"""Calls of several host threads that share a kernel but not its shared-memory
size: f(y), the Jacobian and the LU solve of mechanisms of the same cell shape
and different process counts, each thread on its own stream."""
import json
import threading

import numpy as np
import pytest

from paper_2111_07436_gb300 import camp, workloads as w

pytestmark = pytest.mark.gpu


def _gas(n):
    part = [max(1, round(k * n / 72)) for k in (112, 28, 28, 9, 9)]
    return w.gas_mechanism(f"gas-{n}", n, *part, seed=1000 + n)


# large batches of f(y) share one kernel; cells of up to 32 species share the
# others' one-slot kernels
@pytest.mark.parametrize("mechs,cells", [((w.small_gas_mechanism, w.large_gas_mechanism), 14000),
                                         ((w.small_gas_mechanism, lambda: _gas(32)), 200)])
def test_threads_share_kernels(cuda, mechs, cells):
    import torch
    jobs, errors = [], []
    for i, f in enumerate(mechs):
        mj = f()
        m = camp.Mechanism(json.dumps(mj))
        y, env = (torch.tensor(a, device=cuda) for a in w.cells(mj, cells, seed=i))
        b = torch.ones_like(y)
        calls = [lambda m=m, y=y, env=env, s=None: m.forcing(y, env, stream=s)]
        if cells < 1000:
            calls += [lambda m=m, y=y, env=env, s=None: m.jacobian(y, env, stream=s),
                      lambda m=m, y=y, env=env, b=b, s=None: m.lu_solve(y, env, 0.1, b, stream=s)[0]]
        jobs.append([(c, c()) for c in calls])
    torch.cuda.synchronize()
    start = threading.Barrier(2 * len(jobs))

    def work(job):
        try:
            s = torch.cuda.Stream()
            with torch.cuda.stream(s):
                start.wait()
                got = [c(s=s) for _ in range(150) for c, _ in job]
            s.synchronize()
            for i, g in enumerate(got):
                if not torch.equal(g, job[i % len(job)][1]):
                    errors.append("another result")
        except Exception as e:  # noqa: BLE001
            errors.append(repr(e))
            start.abort()

    threads = [threading.Thread(target=work, args=(job,)) for job in jobs for _ in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[:3]
