"""Launch shapes that the library chooses by size: the results must not depend on the choice.

Every comparison is bit for bit: a work item runs the same arithmetic whichever templates share it.
"""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def _spectrum(n, seed):
    import torch

    return torch.from_numpy(synth.complex_noise(np.random.default_rng(seed), n).astype(np.complex64)).cuda()


@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("n,n_temp", [(1, 85), (1629, 85), (4099, 9), (65536, 85), (200003, 43), (500001, 127)])
def test_chosen_templates_per_item_equal_one_item_per_segment(n, n_temp, prec):
    import torch

    import paper_1806_01556_gb300 as fd

    p = fd.Params(n_temp=n_temp, z_min=-(n_temp // 2), precision=prec)
    s = fd.Searcher(p, n)
    spec = _spectrum(n, n)
    s.plane.fill_(-1.0)
    fd.fdas_convolve(p, spec, n, s.tmpl, s.plane, s.ld)
    got = s.plane.clone()
    s.plane.fill_(-1.0)
    fd.fdas_convolve_cfg(p, spec, n, s.tmpl, s.plane, s.ld, 0, n_temp)
    torch.cuda.synchronize()
    assert torch.equal(got, s.plane)
    assert (got[:, :n] >= 0).all()
