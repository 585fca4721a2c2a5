"""Maxwellian tails below the smallest normal FP32 number on ragged velocity grids (nv % 4 != 0):
a gas at rest at Kn 1e-4, where three steps replace f almost wholly by the Maxwellian of its
moments, keeps its subnormal values as the FP64 oracle does.  M between 1e-41 and 1.1e-38 is
held to one part in 7000 (spacing 1.4e-45); the exponent's FP32 rounding (130 x 2^-24) and the
error of T (1e-6 x 90) add less than 2e-4: within 1e-3."""
import numpy as np
import pytest

import bgk_inputs as bi
import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2408_02350_gb300 import _build
    _build.build()
    import paper_2408_02350_gb300 as g
    return g


@pytest.mark.parametrize("nv", [26, 27])
@pytest.mark.parametrize("order", [1, 2])
def test_subnormal_tails_survive_the_relaxation(g, nv, order):
    p = bi.config("cavity2d_n41_v16_f64", n=11, nv=nv, vmax=14.0, storage="f32", kn=1e-4, time_order=order,
                  lid_u=[0.0, 0.0, 0.0])
    cl = bi.cloud_for(p)
    M = oracle.maxwellian(p, 1.0, (0.0, 0.0), 1.0)
    tail = (M > 1e-41) & (M < 1.1e-38)
    assert tail.sum() >= 8
    sim = oracle.Simulation(p, cl)
    sim.run(3)
    inner = cl["kind"] == 0
    want = sim.f.reshape((-1,) + M.shape)[inner][:, tail]
    s = g.Solver([p], [cl])
    s.set_maxwellian()
    s.step(3)
    s.sync()
    f = s.get_f(0, np.float64).reshape((-1,) + M.shape)[inner][:, tail]
    s.close()
    assert np.abs(f / want - 1.0).max() < 1e-3
