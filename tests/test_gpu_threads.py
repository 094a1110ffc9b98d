"""Handles of several host threads, each with a stream of its own, stepping at
once for the first time in a process: every thread's launches need another
amount of shared memory of the same kernels."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))

PROGRAM = r"""
import sys, threading
sys.path[:0] = [%(root)r, %(here)r]
import numpy as np, torch
import paper_1008_0861_gb300 as P
import workloads as W
from gpu_util import GpuGrid

SIDES = [1100, 1300, 1500, 1700, 1900, 2044]
forms = [dict(prec=p, limiter=l, fp16=f) for p in (1, 0) for l in (0, 1) for f in ((False, True) if p else (False,))]
bad = []
for form in forms:
    sides = SIDES if form["prec"] else [560, 640, 720, 800, 900, 1020]
    # (whole lines, then ragged ones)
    for odd in (0, 1):
        insts = [W.random_instance(n + odd, 64 + odd, seed=n, dt_factor=20.0) for n in sides]
        grids = [GpuGrid(P, i, graph=False, **form) for i in insts]
        streams = [torch.cuda.Stream() for _ in grids]
        for g, s in zip(grids, streams):
            P.aniso_set_option(g.h, P.ANISO_OPT_STREAM, s.cuda_stream)
        torch.cuda.synchronize()
        barrier = threading.Barrier(len(grids))

        def work(g, i):
            barrier.wait()
            try:
                for _ in range(5):
                    P.aniso_step(g.h, g.T, i.dt, 1)
                P.aniso_sync(g.h)
            except Exception as e:
                bad.append((form, i.nx, str(e)))

        threads = [threading.Thread(target=work, args=(g, i)) for g, i in zip(grids, insts)]
        [t.start() for t in threads]
        [t.join() for t in threads]
        alone = [GpuGrid(P, i, graph=False, **form) for i in insts]
        for g, a, i in zip(grids, alone, insts):
            for _ in range(5):
                P.aniso_step(a.h, a.T, i.dt, 1)
            P.aniso_sync(a.h)
            if not torch.equal(g.T, a.T):
                bad.append((form, i.nx, "differs"))
        [g.close() for g in grids + alone]
for b in bad:
    print(b)
sys.exit(1 if bad else 0)
"""


@pytest.mark.parametrize("attempt", range(3))
def test_threads_that_launch_at_once(lib, attempt):
    program = PROGRAM % {"root": os.path.dirname(HERE), "here": HERE}
    r = subprocess.run([sys.executable, "-c", program], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-2000:]
