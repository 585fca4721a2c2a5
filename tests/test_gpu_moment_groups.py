"""The moments that bgk_set_f takes, at every number of points per warp (1, 2 and 4 by the size
of the cloud) and of warps per CTA, with clouds that leave the last CTA partly filled: rho, U
and T of every point against FP64 sums of the stored values.  The kernel rounds a term at most
six times in FP32 (node, products, sums of four) and compensates the rest, so a sum is within
6 x 2^-24 of the sum of its terms' magnitudes: 1e-6 for rho, 3e-6 for U (mean |v| below 3) and
T."""
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


@pytest.mark.parametrize("storage", ["f32", "bf16"])
@pytest.mark.parametrize("dim,n,nv", [(2, 3, 4), (2, 41, 5), (2, 101, 4), (2, 101, 5), (2, 151, 4), (2, 151, 13),
                                      (2, 181, 5), (2, 211, 4), (3, 5, 3), (3, 21, 3), (3, 21, 4), (3, 31, 5)])
def test_moments_of_every_point(g, storage, dim, n, nv):
    import torch
    p = bi.config("cavity2d_n41_v16_f64" if dim == 2 else "cavity3d_n41_v16_f32", n=n, nv=nv, vmax=3.0, storage=storage)
    M = oracle.maxwellian(p, 1.0, (0.1, -0.05, 0.02)[:dim], 1.0)
    u = bi.uniform01(3, n ** dim * M.size).reshape((-1,) + M.shape)
    f = torch.from_numpy(M[None] * (0.8 + 0.4 * u)).to({"f32": torch.float32, "bf16": torch.bfloat16}[storage]).cuda()
    s = g.Solver([p], [bi.cloud_for(p)])
    s.set_f(f)
    rho, U, T = s.moments()
    s.close()
    h = f.double().cpu().numpy()
    v = oracle.velocity_grid(dim, nv, 3.0).reshape(-1, dim)
    R = h[:, 0].sum(1)
    Uw = h[:, 0] @ v / R[:, None]
    E = h[:, 0] @ (v * v).sum(1) + (h[:, 1].sum(1) if dim == 2 else 0.0)
    Tw = (E / R - (Uw * Uw).sum(1)) / 3.0
    wv = oracle.dv(nv, 3.0) ** dim
    assert np.abs(rho / (R * wv) - 1.0).max() < 1e-6
    assert np.abs(U - Uw).max() < 3e-6 and np.abs(T - Tw).max() < 3e-6
