"""The branches of the FP64 transport against the oracle's FP64 step: mirror-paired chunks
(nv % 4 == 0, fixed points), row chunks (ALE), ragged grids (nv % 4 != 0), more chunks than
threads of a CTA (NV = 2304, 1728 and 4096), the smallest pairable grid, two stages with
averaging.  Both sides sum about 20 (80) products per velocity and NV products per moment
in FP64, so they agree to NV times 2^-53 with a wide margin at 1e-11.
"""
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


@pytest.mark.parametrize("dim,n,nv,ale,order", [
    (2, 9, 4, 0, 1), (2, 11, 48, 0, 1), (2, 11, 48, 1, 1), (2, 9, 47, 0, 1), (2, 9, 47, 1, 1), (2, 9, 12, 0, 2),
    (3, 6, 4, 0, 1), (3, 5, 12, 1, 1), (3, 5, 16, 0, 1), (3, 5, 7, 0, 2)])
def test_fp64_transport_branches_match_the_oracle(g, dim, n, nv, ale, order):
    name = "cavity2d_n41_v16_f64" if dim == 2 else "cavity3d_n41_v16_f32"
    p = bi.config(name, n=n, nv=nv, vmax=3.0, storage="f64", ale=ale, time_order=order)
    cl = bi.cloud_for(p)
    nc = 2 if dim == 2 else 1
    M = oracle.maxwellian(p, 1.0, (0.1, -0.05, 0.02)[:dim], 1.0)
    u = bi.uniform01(5, len(cl["kind"]) * M.size).reshape((-1,) + M.shape)
    f0 = np.ascontiguousarray(M[None] * (1.0 + 0.1 * (2.0 * u - 1.0)))
    assert f0.shape == (len(cl["kind"]), nc, nv ** dim)
    sim = oracle.Simulation(p, cl, f0=f0)
    sim.run(2)
    s = g.Solver([p], [cl])
    s.set_f(f0)
    s.step(2)
    s.sync()
    f = s.get_f(0, np.float64)
    rho, U, T = s.moments()
    s.close()
    assert np.abs(f - sim.f).max() < 1e-11 * np.abs(sim.f).max()
    assert np.abs(rho - sim.rho).max() < 1e-11 and np.abs(U - sim.U).max() < 1e-11 and np.abs(T - sim.T).max() < 1e-11
