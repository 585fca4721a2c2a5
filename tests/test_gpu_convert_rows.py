"""Uploads and read-backs of f between padded and dense rows, below and above 256 elements per
row (blocks of rows of 4096 elements, a warp per row): rows of 9 to 6859 velocities, more and
fewer rows than a block holds, blocks filled exactly and in part.  Values survive the round trip through the padded storage exactly,
and each element lands at its own place (every value is distinct)."""
import numpy as np
import pytest

import bgk_inputs as bi

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


@pytest.mark.parametrize("dim,n,nv", [(2, 3, 3), (2, 15, 3), (2, 60, 3), (2, 16, 5), (2, 31, 11), (2, 9, 15), (2, 9, 17), (2, 7, 45),
                                      (2, 4, 63),
                                      (3, 3, 3), (3, 7, 5), (3, 5, 13), (3, 3, 19)])
def test_padded_rows_round_trip(g, dim, n, nv):
    import torch
    p = bi.config("cavity2d_n41_v16_f64" if dim == 2 else "cavity3d_n41_v16_f32", n=n, nv=nv, vmax=3.0, storage="f64")
    s = g.Solver([p], [bi.cloud_for(p)])
    shape = (n ** dim, 2 if dim == 2 else 1, nv ** dim)
    f = (1.0 + torch.arange(int(np.prod(shape)), dtype=torch.float64).reshape(shape) / 2 ** 22).cuda()
    s.set_f(f)
    out = torch.zeros_like(f)
    g.bgk_get_f(s.ctx, 0, out, g.BGK_F64)
    assert torch.equal(out, f)
    out32 = torch.zeros(shape, dtype=torch.float32, device="cuda")
    g.bgk_get_f(s.ctx, 0, out32, g.BGK_F32)
    assert torch.equal(out32, f.float())
    s.close()
