"""The range-checked build on meshes large enough for the kernels with one element per lane: the acoustic tile kernels with the
projection inside and apart, FP32 and FP64, their adjoint forms, and the elastic ones, each with a ragged last tile and every
face orientation. No index out of range, and the normal build's results."""
import os
import subprocess
import sys
import textwrap

import numpy as np
import pytest

from paper_1808_08645_gb300 import build as libbuild
from parity_util import TOL_STAGE, rel_l2

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CASES = textwrap.dedent("""
    import sys, numpy as np
    sys.path.insert(0, {root!r})
    from paper_1808_08645_gb300 import binding as B, inputs
    lib = {lib!r}
    if lib:
        B.lib_path = lambda: lib
    out = {{}}
    n3 = lambda n: (n + 1) * (n + 2) * (n + 3) // 6
    mesh = lambda h: inputs.cube_mesh(h, jitter=0.1, shuffle=True, seed=h)
    for N, h, prec in ((2, 13, 32), (3, 12, 32), (6, 24, 32), (5, 10, 64)):
        v, e = mesh(h)
        rng = np.random.default_rng(N)
        s = B.Solver(v, e, N, 1, prec)
        s.set_c2(rng.uniform(0.5, 2.0, (len(e), 4)))
        s.set_state(rng.standard_normal((4, len(e), n3(N))))
        s.step(1e-4, 1)
        s.sync()
        out["acoustic%d" % N] = s.get_state()[0]
        s.close()
    v, e = mesh(7)
    s = B.Solver(v, e, 5, 2, 32)
    s.set_state(np.random.default_rng(5).standard_normal((4, len(e), 56)))
    s.set_receivers([[0.3, 0.4, 0.5], [0.7, 0.6, 0.2]])
    s.set_point_source([0.5, 0.5, 0.5], B.ricker_samples(1e-4, 2, f0=10.0, t0=0.05))
    s.record(1e-4, 2, 1)
    gc, gq = s.adjoint(np.ones((2, 2)), want_q0=True)
    out["gc"], out["gq"] = gc, gq
    s.close()
    for N, h in ((2, 15), (3, 14), (5, 11), (6, 11), (7, 7)):
        v, e = mesh(h)
        s = B.ElasticSolver(v, e, N, 2, 32)
        s.set_media(*inputs.elastic_media(v, e, 2))
        s.set_state(np.random.default_rng(N).standard_normal((9, len(e), n3(N))))
        s.step(1e-4, 1)
        s.sync()
        out["elastic%d" % N] = s.get_state()[0]
        s.close()
    np.savez({path!r}, **out)
""")


def run(tmp_path, lib, name):
    path = str(tmp_path / f"{name}.npz")
    script = tmp_path / f"{name}.py"
    script.write_text(CASES.format(root=ROOT, lib=lib, path=path))
    p = subprocess.run([sys.executable, str(script)], capture_output=True, text=True, timeout=900)
    assert p.returncode == 0, p.stderr[-2000:]
    return np.load(path)


def test_checked_build_runs_the_lane_kernels_clean_and_agrees(tmp_path):
    checked = libbuild.build(checked=True)
    libbuild.build()
    got, want = run(tmp_path, checked, "checked"), run(tmp_path, "", "normal")
    assert sorted(got.files) == sorted(want.files)
    for k in want.files:
        assert rel_l2(got[k], want[k]) <= TOL_STAGE[32], k
