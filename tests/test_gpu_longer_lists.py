"""3D neighbour lists in arrays of more than 160 entries, of which the FP32 transport stages 160
(the rest are read from global memory): interior points with up to 122 (all staged) and with
more than 160 neighbours, through the mirror-paired, the aligned, the ragged and the ALE
kernels, against the FP64 oracle within the project's FP32 bar of 1e-4."""
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


@pytest.mark.parametrize("cap,radius,least", [(161, 3.05, 100), (320, 3.7, 165), (512, 3.7, 165)])
@pytest.mark.parametrize("nv,ale", [(8, 0), (6, 0), (8, 1), (6, 1)])
def test_lists_in_long_arrays(g, cap, radius, least, nv, ale):
    p = bi.config("cavity3d_n41_v16_f32", n=10, nv=nv, vmax=3.0, ale=ale, max_nbrs=cap)
    p["h"] = radius * p["dx"]
    cl = bi.cloud_for(p)
    cnt, _ = oracle.neighbours(cl["x"], p["h"], cap=cap)
    assert cnt[cl["kind"] == 0].max() > least
    sim = oracle.Simulation(p, cl)
    sim.run(2)
    s = g.Solver([p], [cl])
    s.set_maxwellian()
    s.step(2)
    s.sync()
    rho, u, T = s.moments()
    f = s.get_f(0, np.float64)
    s.close()
    assert np.abs(rho - sim.rho).max() < 1e-4 and np.abs(T - sim.T).max() < 1e-4 and np.abs(u - sim.U).max() < 1e-4
    assert np.abs(f - sim.f).max() < 1e-4 * np.abs(sim.f).max()
