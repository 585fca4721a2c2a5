"""The side chain of moving-point steps (motion, lists and stencils of the next step as one
cooperative launch): contexts of different sizes side by side."""
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
