"""The branches of the FP32 adjoint kernels (aligned and ragged velocity grids, 2D and 3D, no
collisions) against the oracle's adjoint step, from a non-uniform state and a random adjoint
field.  FP32 sums of at most 80 products per velocity and of NV terms per point: 2e-4 of the
largest entry, the bar of the project's FP32 gradients."""
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


@pytest.mark.parametrize("dim,n,nv,tau_mode", [
    (2, 11, 8, 0), (2, 11, 7, 0), (2, 9, 13, 1), (2, 9, 12, 2), (3, 6, 4, 0), (3, 6, 5, 0)])
def test_fp32_adjoint_branches_match_the_oracle(g, dim, n, nv, tau_mode):
    import torch
    name = "adjoint2d_n101_v24_f32" if dim == 2 else "cavity3d_n41_v16_f32"
    p = bi.config(name, n=n, nv=nv, vmax=3.0, storage="f32", tau_mode=tau_mode)
    cl = bi.cloud_for(p)
    M = oracle.maxwellian(p, 1.0, (0.1, -0.05, 0.02)[:dim], 1.0)
    npts, NV = len(cl["kind"]), nv ** dim
    u = bi.uniform01(7, 2 * npts * M.size).reshape((2, npts) + M.shape)
    f = np.ascontiguousarray((M[None] * (1.0 + 0.1 * (2.0 * u[0] - 1.0))).astype(np.float32).astype(np.float64))
    lam = np.ascontiguousarray((2.0 * u[1] - 1.0).astype(np.float32).astype(np.float64))
    cnt, col = oracle.neighbours(cl["x"], p["h"], cap=p["max_nbrs"])
    st = oracle.stencils(p, cl["x"], cl["kind"], cnt, col)
    want, dth = oracle.adjoint_step(p, cl["kind"], cl["normal"], cnt, col, st, f, lam)
    s = g.Solver([p], [cl])
    s.set_f(f.astype(np.float32))
    nvp = s.stats()["nv_pad"]
    lin = torch.zeros((npts, M.shape[0], nvp), dtype=torch.float32, device="cuda")
    lin[..., :NV] = torch.from_numpy(lam.astype(np.float32)).cuda()
    lout = torch.full_like(lin, float("nan"))
    th = torch.zeros(4, dtype=torch.float64, device="cuda")
    g.bgk_adjoint_step(s.ctx, 0, lin, lout, th)
    s.sync()
    got = lout[..., :NV].double().cpu().numpy()
    s.close()
    assert np.abs(got - want).max() < 2e-4 * np.abs(want).max()
    if tau_mode != 2:
        assert abs(float(th[3]) - dth[3]) < 2e-4 * max(abs(dth[3]), np.abs(dth).max())
