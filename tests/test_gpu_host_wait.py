"""A solve's host thread waits for the device the way its process asked the CUDA runtime to."""
import json
import pathlib
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

# CPU seconds and wall seconds of a solving thread, in a process that set its device's schedule flags
RUN = """
import ctypes, json, sys, time
flags = int(sys.argv[1])
cu = ctypes.CDLL("libcuda.so.1")
assert cu.cuInit(0) == 0
assert cu.cuDevicePrimaryCtxSetFlags_v2(0, flags) == 0
import torch
import paper_2401_09961_gb300 as irls
X = torch.randn(2048, 2048, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
with irls.Plan(2048, 2048, precision="bf16x3", tau=1e-2, delta=1e-3, outer_iters=2, cg_tol=0.0,
               cg_max_iter=400) as p:
    p.unwrap(X)
    runs = []
    for _ in range(3):
        c, t = time.thread_time(), time.perf_counter()
        U, st = p.unwrap(X)
        runs.append([time.perf_counter() - t, time.thread_time() - c, sum(st["cg_iters"])])
    print("TIMES", json.dumps(min(runs)))
"""


def times(flags):
    r = subprocess.run([sys.executable, "-c", RUN, str(flags)], capture_output=True, text=True,
                       timeout=300, cwd=pathlib.Path(__file__).resolve().parents[1])
    assert r.returncode == 0, r.stderr[-2000:]
    return json.loads(r.stdout.split("TIMES", 1)[1])


def test_blocking_waits_leave_the_core():
    """CU_CTX_SCHED_BLOCKING_SYNC (4): a wait of four iterations (1 ms at 2048^2) sleeps; what is left
    is the launches, about 5 a 250 us iteration.  A spin takes the whole time."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    wall, cpu, its = times(4)   # the quickest of three runs
    assert its == 800
    assert cpu <= 0.6 * wall, (cpu, wall)
    spin_wall, _, _ = times(1)
    # and the sleeps fit the iterations in flight (a 70 us sleep after every 250 us one: 1.28)
    assert wall <= 1.15 * spin_wall, (wall, spin_wall)
