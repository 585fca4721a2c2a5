"""The side chain of moving-point steps (motion, lists and stencils of the next step as one
cooperative launch): contexts of different sizes side by side, a launch that the runtime
refuses, and a wait that gives up before any list is there."""
import os
import subprocess
import sys

import numpy as np
import pytest

import bgk_inputs as bi

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def g():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2408_02350_gb300 import _build
    _build.build()
    import paper_2408_02350_gb300 as g
    return g


def _ale(**over):
    return bi.config("cavity2d_ale_n201_v32_f32", **dict(dict(n=21, nv=8, vmax=4.0), **over))


@pytest.mark.parametrize("wls", [1, 2])
def test_contexts_with_different_candidate_capacities_step_in_turn(g, wls):
    # skin = h: 2253 and 1760 candidates per point, 72 and 56 KB of shared memory per CTA;
    # the smaller context must not lower the larger one's limit.  Each steps as it does alone.
    ps = [_ale(wls_order=wls, skin=1.0, max_nbrs=cap) for cap in (512, 400)]
    alone = []
    for p in ps:
        s = g.Solver([p], [bi.cloud_for(p)])
        s.set_maxwellian()
        s.step(6)
        s.sync()
        alone.append((s.get_f(0, np.float32), s.positions()))
        s.close()
    both = [g.Solver([p], [bi.cloud_for(p)]) for p in ps]
    for s in both:
        s.set_maxwellian()
    for _ in range(3):
        for s in both:
            s.step(2)
    for s, (f, x) in zip(both, alone):
        s.sync()
        assert np.array_equal(s.get_f(0, np.float32), f) and np.array_equal(s.positions(), x)
        s.close()


# The cases below step in a process of their own (argv: library, output folder).
_REFUSED = [{"wls_order": 1}, {"wls_order": 2}, {"wls_order": 2, "storage": "bf16"}, {"body": True, "n": 41}]
_STEP = r"""
import sys
import numpy as np
sys.path.insert(0, %(root)r)
import bgk_inputs as bi
import paper_2408_02350_gb300 as g
g.LIB_PATH = sys.argv[1]
for k, over in enumerate(%(cases)r):
    over = dict(over)
    name = "body2d_ale_n201_v32_f32" if over.pop("body", False) else "cavity2d_ale_n201_v32_f32"
    p = bi.config(name, **dict(dict(n=21, nv=8, vmax=4.0), **over))
    s = g.Solver([p], [bi.cloud_for(p)])
    s.set_maxwellian()
    s.step(5)
    s.sync()
    np.savez(sys.argv[2] + "/%%d.npz" %% k, f=s.get_f(), x=s.positions(), n=s.stats()["launches"])
    s.close()
"""


def test_a_refused_cooperative_launch_falls_back_to_the_separate_kernels(g, tmp_path):
    # a build whose cooperative grid is 64 times what fits: the runtime refuses the launch
    # (an error code, nothing runs); the separate kernels then give the same bits
    from paper_2408_02350_gb300 import _build
    big = _build._build_into(str(tmp_path / "build"), str(tmp_path / "libbgk_big.so"), False, False,
                             ["-DBGK_CHAIN_GRID_SCALE=64"])
    for tag, lib in (("a", _build.lib_path()), ("b", big)):
        os.makedirs(str(tmp_path / tag))
        r = subprocess.run([sys.executable, "-c", _STEP % {"root": ROOT, "cases": _REFUSED}, lib, str(tmp_path / tag)],
                           capture_output=True, text=True, timeout=600)
        assert r.returncode == 0, r.stderr[-2000:]
    for k in range(len(_REFUSED)):
        a, b = np.load(str(tmp_path / ("a/%d.npz" % k))), np.load(str(tmp_path / ("b/%d.npz" % k)))
        assert np.array_equal(a["f"], b["f"]) and np.array_equal(a["x"], b["x"]), k
        assert b["n"] > a["n"], k


@pytest.mark.parametrize("wls,storage", [(1, "f32"), (2, "f32"), (2, "bf16")])
def test_timeout_on_the_first_step_is_reported_as_such(g, wls, storage):
    # one poll per wait: the rows of the next step's lists that no CTA reached are empty,
    # and their stencils and wall weights singular in consequence; the run then continues
    # as one without a timeout
    p = _ale(wls_order=wls, storage=storage, n=41)
    ref = g.Solver([p], [bi.cloud_for(p)])
    ref.set_maxwellian()
    ref.step(6)
    ref.sync()
    s = g.Solver([p], [bi.cloud_for(p)])
    s.set_maxwellian()
    g.bgk_set_watchdog(s.ctx, 1)
    s.step(1)
    with pytest.raises(g.BGKError) as e:
        s.sync()
    assert e.value.code == g.BGK_E_TIMEOUT
    g.bgk_set_watchdog(s.ctx, 0)
    s.step(5)
    s.sync()
    assert np.array_equal(s.get_f(), ref.get_f()) and np.array_equal(s.positions(), ref.positions())
    s.close()
    ref.close()


# Second-order stencils on moving points: lists from the side chain, the fit after it.  FP32
# within the project's 1e-4; BF16 rounds f once per step to 2^-9, so three steps are within
# 3 x 2^-9 of rho and T (6e-3) even if every rounding had the same sign.
@pytest.mark.parametrize("dim,n,nv,storage,body,steps,tol", [
    (3, 9, 6, "f32", False, 6, 1e-4), (3, 9, 8, "f32", False, 6, 1e-4), (3, 9, 6, "bf16", False, 3, 6e-3),
    (2, 21, 8, "bf16", False, 3, 6e-3), (2, 21, 7, "bf16", False, 3, 6e-3), (2, 41, 8, "f32", True, 8, 1e-4)])
def test_second_order_stencils_of_moving_points(g, dim, n, nv, storage, body, steps, tol):
    import oracle
    name = "body2d_ale_n201_v32_f32" if body else "cavity2d_n41_v16_f64" if dim == 2 else "cavity3d_n41_v16_f32"
    p = bi.config(name, n=n, nv=nv, vmax=4.0, storage=storage, ale=1, wls_order=2)
    cl = bi.cloud_for(p)
    sim = oracle.Simulation(p, cl)
    sim.run(steps)
    s = g.Solver([p], [cl])
    s.set_maxwellian()
    s.step(steps)
    s.sync()
    rho, u, T = s.moments()
    x = s.positions()
    s.close()
    assert np.abs(rho - sim.rho).max() < tol * np.abs(sim.rho).max() and np.abs(T - sim.T).max() < tol * np.abs(sim.T).max()
    if storage == "f32":
        assert np.abs(u - sim.U).max() < tol * np.abs(sim.U).max() and np.abs(x - sim.x).max() < 1e-6


def test_second_order_stencils_of_moving_points_in_slabs(g):
    # two velocity slabs of the same case, the same bar against the oracle
    import oracle
    from paper_2408_02350_gb300.sharded import ShardedSolver
    p = _ale(wls_order=2)
    cl = bi.cloud_for(p)
    sim = oracle.Simulation(p, cl)
    sim.run(6)
    s = ShardedSolver.on_one_device(p, cl, 2)
    s.set_maxwellian()
    s.step(6)
    s.sync()
    rho, u, T = s.moments()
    assert np.abs(rho - sim.rho).max() < 1e-4 and np.abs(u - sim.U).max() < 1e-4 and np.abs(T - sim.T).max() < 1e-4
