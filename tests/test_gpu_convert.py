"""Uploads and read-backs of f at the edges of the copy kernels (flat copies of whole arrays
when NV % 4 == 0 and the pointers are aligned, row copies otherwise): every pair of caller
and storage types, ragged rows, a misaligned device tensor, and point counts below and
above one group of points of the moments kernel.  The conversions are exact or one
rounding, the same as torch's."""
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


@pytest.mark.parametrize("storage", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("n,nv", [(5, 2), (7, 3), (9, 8), (75, 5)])
@pytest.mark.parametrize("offset", [0, 1])
def test_set_f_and_get_f_convert_every_element(g, storage, n, nv, offset):
    import torch
    dt = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16}
    code = {"f64": g.BGK_F64, "f32": g.BGK_F32, "bf16": g.BGK_BF16}
    p = bi.config("cavity2d_n41_v16_f64", n=n, nv=nv, vmax=3.0, storage=storage)
    s = g.Solver([p], [bi.cloud_for(p)])
    count = n * n * 2 * nv * nv
    gen = torch.Generator().manual_seed(3)
    for src in dt:
        whole = torch.rand(count + offset, generator=gen, dtype=torch.float64).add(0.5).to(dt[src]).cuda()
        x = whole[offset:]
        g.bgk_set_f(s.ctx, 0, x, code[src])
        held = x.to(torch.float32 if src == "f64" and storage == "bf16" else dt[src]).to(dt[storage])
        rho, _, _ = s.moments()
        want = held.double().reshape(n * n, 2, nv * nv)[:, 0].sum(1).cpu().numpy() * (6.0 / (nv - 1)) ** 2
        assert np.abs(rho - want).max() < 1e-6 * want.max()
        for dst in dt:
            out = torch.zeros(count + offset, dtype=dt[dst], device="cuda")
            g.bgk_get_f(s.ctx, 0, out[offset:], code[dst])
            back = held.to(torch.float32 if storage == "f64" and dst == "bf16" else dt[storage]).to(dt[dst])
            assert torch.equal(out[offset:], back), (src, dst)
    s.close()
