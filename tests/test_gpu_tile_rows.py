"""Tile shapes that a caller sets are the ones that run, on small images too; the default stands for
the library's choice, and the autotuner times a launch once."""
import json
import pathlib
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def irls():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2401_09961_gb300 as m
    m.lib()
    return m


OPTS = dict(tau=1e-2, delta=1e-3, outer_iters=1, cg_tol=1e-6, cg_max_iter=3)

# the grids of the direction and update launches of a solve at each tile shape, from a trace of a
# process of its own
TRACE = """
import json, sys
import torch
import paper_2401_09961_gb300 as irls
h, w, prec, shapes, path = json.loads(sys.argv[1])
X = torch.randn(h, w, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
out = []
with irls.Plan(h, w, precision=prec, tau=1e-2, delta=1e-3, outer_iters=1, cg_tol=1e-6,
               cg_max_iter=3) as p:
    for s in shapes[:1] + shapes:   # (the first trace of a process is empty)
        p.set_tiles(*s)
        with torch.profiler.profile() as t:
            p.unwrap(X)
            torch.cuda.synchronize()
        t.export_chrome_trace(path)
        seen = {}
        for e in json.load(open(path))["traceEvents"]:
            for k in ("k_direction_pap", "k_update"):
                if e.get("cat") == "kernel" and k in e.get("name", ""):
                    seen.setdefault(k, set()).add(e["args"]["grid"][1])
        out.append({k: sorted(v) for k, v in seen.items()})
print("GRIDS", json.dumps(out[1:]))
"""


@pytest.mark.parametrize("prec", ["fp32", "bf16x3"])
def test_set_rows_hold_on_small_images(irls, prec, tmp_path):
    """203 x 613, where one wave is a row a block: the default takes it, a set count holds."""
    shapes = [(24, 32), (8, 8), (16, 24), (32, 16), (22, 27)]
    arg = json.dumps([203, 613, prec, shapes, str(tmp_path / "trace.json")])
    r = subprocess.run([sys.executable, "-c", TRACE, arg], capture_output=True, text=True,
                       timeout=300, cwd=pathlib.Path(__file__).resolve().parents[1])
    assert r.returncode == 0, r.stderr[-2000:]
    out = json.loads(r.stdout.split("GRIDS", 1)[1])
    if not all(out):
        pytest.skip("no kernel trace on this machine")
    assert out[0] == {"k_direction_pap": [203], "k_update": [203]}
    for (d, u), got in zip(shapes[1:], out[1:]):
        assert got == {"k_direction_pap": [-(-203 // d)], "k_update": [-(-203 // u)]}, (d, u)


def test_autotune_times_a_launch_once(irls):
    """1030 x 2050: the defaults take one wave's rows, which are among the other candidates of the
    direction or update kernel or not; equal launches report equal times, so the first is kept."""
    with irls.Plan(1030, 2050, precision="bf16x3", **OPTS) as p:
        ms = p.autotune()["ms"]
        rows = (8, 16, 24, 32)
        if p.tiles[0] in rows:
            assert p.tiles[0] == rows[int(np.argmin(ms[:4]))]
        if p.tiles[1] in rows:
            assert p.tiles[1] == rows[int(np.argmin(ms[4:]))]
    with irls.Plan(2048, 2048, precision="bf16x3", **OPTS) as p:
        p.autotune()
        # the one-wave counts at this size are the defaults' launches, not candidates of their own
        assert all(t in (8, 16, 24, 32) or t > 32 for t in p.tiles), p.tiles
