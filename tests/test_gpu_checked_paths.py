"""The checked build (every kernel index tested against its range) over the paths that
small and special handles take: FP64 blocks shared by 8, 4 and 2 CTAs (1, 18, 34 and
48 blocks; resolution changes, refluxing, a background field, the body, local time
steps), every kind of background field in both forms, items of several blocks, and
states loaded and stored whole and per grid.  No index may leave its range, and the
checked library must give the normal library's results (FP64 to 1e-12, mixed to 1e-5
of a variable's largest value).  The checked runs happen in a child process (one
library per process, chosen by BATS_LIB)."""
import os
import subprocess
import sys

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, os.path.dirname(HERE))


def _grid(root, refine, bc, **more):
    from paper_2501_06717_gb300 import workloads as W
    lo, hi = (-1.0,) * 3, (1.0,) * 3
    leaves = W.uniform_leaves(root)
    if refine:
        leaves = W.balance(W.refine_where(leaves, lambda b0, b1: bool(np.all(b0 <= 0.0) and np.all(b1 >= 0.0)), lo, hi,
                                          root, 1), root, (bc == W.BC_PERIODIC,) * 3)
    prob = W.Problem("checked", lo, hi, root, W.as_leaf_array(W.morton_sort(leaves)), (bc,) * 6, **more)
    x = W.cell_centres(lo, hi, root, prob.leaves)
    s = [np.sin(np.pi * (a + 0.1 * k)) for k, a in enumerate(x)]
    w = [1 + 0.3 * s[0] * s[1], 0.5 * s[1], 0.4 * s[2], 0.3 * s[0], 0.5 * s[2], 0.4 * s[0], 0.6 + 0.2 * s[1], 1 + 0.3 * s[2]]
    if prob.body_r:
        inside = x[0] * x[0] + x[1] * x[1] + x[2] * x[2] < prob.body_r ** 2
        w = [np.where(inside, prob.body[v], w[v]) for v in range(8)]
    return W.with_state(prob, w)


def _run_all(out_path):
    """Every case through the library that BATS_LIB names; results to an npz."""
    from paper_2501_06717_gb300 import bats as B
    from paper_2501_06717_gb300 import workloads as W
    body = dict(body_r=0.3, body=np.array([1.5, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 1.2]))
    dipole = dict(b0=W.B0_DIPOLE, b0_param=np.array([0.0, 0.0, 0.05] + [0.0] * 9), powell=1)
    linear = dict(b0=W.B0_LINEAR, b0_param=np.array([0.1, 0.2, 0.3, 0.1, 0.02, 0.0, 0.03, -0.1, 0.0, 0.0, 0.01, 0.05]))
    uniform = dict(b0=W.B0_UNIFORM, b0_param=np.array([0.1, 0.2, 0.3] + [0.0] * 9))
    cases = [("one", (1, 1, 1), False, W.BC_PERIODIC, {}), ("one_outflow", (1, 1, 1), False, W.BC_OUTFLOW, {}),
             ("eighteen", (3, 3, 2), False, W.BC_OUTFLOW, dict(limiter=W.LIM_MC, flux=W.FLUX_HLL)),
             ("amr_reflux", (3, 3, 3), True, W.BC_OUTFLOW, dict(flux=W.FLUX_LINDE, reflux=1)),
             ("amr_body_dipole", (3, 3, 3), True, W.BC_OUTFLOW, dict(local_dt=1, **body, **dipole)),
             ("forty_eight", (4, 4, 3), False, W.BC_PERIODIC, dict(rk=W.RK_EULER, limiter=W.LIM_NONE, **uniform)),
             ("linear", (4, 4, 4), False, W.BC_OUTFLOW, dict(rk=W.RK_SSP2, **linear))]
    res = {}
    for prec in (0, 1):
        for name, root, refine, bc, more in cases:
            q = _grid(root, refine, bc, **more)
            with B.Solver(q, precision=prec) as s:
                s.set_state(0, q.U0)
                s.step(2, 0.3)
                res["%s_%d" % (name, prec)] = s.get_state(0)
                s.set_state(0, q.U0)
                res["%s_residual_%d" % (name, prec)] = s.residual(0)
        probs = [_grid((3, 3, 2), False, W.BC_OUTFLOW), _grid((2, 2, 2), False, W.BC_PERIODIC)]
        with B.Solver(probs, precision=prec) as s:
            U = np.concatenate([np.ascontiguousarray(p.U0).reshape(-1) for p in probs])
            B.bats_set_states(s.h, U)
            s.step(1, 0.3)
            res["states_%d" % prec] = B.bats_get_states(s.h, np.zeros_like(U)).reshape(1, -1)
    q = _grid((5, 7, 71), False, W.BC_OUTFLOW)
    with B.Solver(q, precision=1, blocks_per_cta=2) as s:
        s.set_state(0, q.U0)
        s.step(1, 0.3)
        res["items_1"] = s.get_state(0)
    np.savez(out_path, **res)


@pytest.mark.gpu
def test_checked_build_on_small_and_special_handles(tmp_path):
    from paper_2501_06717_gb300 import build as BLD
    lib = BLD.build(checked=True)
    paths = {k: str(tmp_path / (k + ".npz")) for k in ("normal", "checked")}
    env = dict(os.environ)
    env.pop("BATS_LIB", None)
    subprocess.run([sys.executable, __file__, paths["normal"]], check=True, env=env, timeout=1200)
    env["BATS_LIB"] = lib
    r = subprocess.run([sys.executable, __file__, paths["checked"]], env=env, timeout=1800, capture_output=True, text=True)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]
    ref, chk = np.load(paths["normal"]), np.load(paths["checked"])
    assert sorted(ref.files) == sorted(chk.files)
    for k in ref.files:
        a, b = ref[k], chk[k]
        a, b = a.reshape(a.shape[0], -1), b.reshape(b.shape[0], -1)
        scale = np.abs(a).max(1)
        for c in ((1, 2, 3), (4, 5, 6)) if len(scale) == 8 else ():
            scale[list(c)] = scale[list(c)].max()
        scale = np.where(scale > 0, scale, 1.0)
        assert (np.abs(a - b).max(1) / scale).max() <= (1e-12 if k.endswith("_0") else 1e-5), k


if __name__ == "__main__":
    _run_all(sys.argv[1])
