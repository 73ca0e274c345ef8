"""The analysis entry points on one context: their kept work memory and their kernels at the sizes
where tiles, line groups and radices end, against the oracle."""
import math

import numpy as np
import pytest

from oracle import diag as odiag
from oracle import isosurface as oiso
from paper_1404_0959_gb300.inputs import random_fields, smooth_field

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fe():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1404_0959_gb300 import build
    build.build()
    from paper_1404_0959_gb300 import fe as fe_mod
    return fe_mod


def test_les_keeps_the_surface_memory(fe):
    """The a-priori LES call between two extractions of one context leaves the second one's work memory alone."""
    import torch
    N = 24
    f = smooth_field(N, 5, 1.0)
    T, _ = oiso.extract(f, 0.1, 2 * math.pi / N)
    s = fe.Solver([dict(N=N, tau_p=[], Y0=[])])
    s.init_state()
    fd = torch.as_tensor(f, device="cuda").contiguous()
    tri = torch.zeros((len(T), 9), dtype=torch.float64, device="cuda")
    n0, a0 = fe.fe_isosurface(s.ctx, 0, fd.data_ptr(), 0.1, tri.data_ptr(), len(T))
    fe.fe_les_apriori(s.ctx, 0, 2, 0.17)
    other = torch.full((64 * N ** 3,), 7.0, device="cuda")  # takes memory that was given back by mistake
    n1, a1 = fe.fe_isosurface(s.ctx, 0, fd.data_ptr(), 0.1, tri.data_ptr(), len(T))
    assert n0 == n1 == len(T) and a0 == a1
    assert float(other.min()) == 7.0 and float(other.max()) == 7.0
    assert np.array_equal(tri.cpu().numpy().reshape(-1, 3, 3), T)
    s.close()
