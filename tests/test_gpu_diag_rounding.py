"""The Gauss residual of a grid without particles is its div E, bit for bit as
differences over cell sizes: a curl's divergence is all rounding, so a quotient
taken in another way shows."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1101_0809_gb300 import build as B
    B.build()
    from paper_1101_0809_gb300 import pic
    return pic


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("dims,n,d", [(2, (19, 14, 1), (0.3, 0.7, 1.0)), (3, (13, 15, 11), (0.3, 0.7, 1.1)),
                                      (3, (13, 15, 11), (0.5, 2.0, 1.0)), (2, (19, 14, 1), (0.25, 0.7, 1.0))])
def test_residual_is_the_divergence_of_e(P, prec, dims, n, d):
    g = P.Grid(P.make_desc(dims, n, d, 0.01, 9.0, prec, tile=(4, 4, 4), halo=0))
    rng = np.random.Generator(np.random.PCG64(88))
    B = [rng.normal(size=g.shape) for _ in range(3)]
    g.set_fields([np.zeros(g.shape)] * 3, B)
    assert P.pic_diagnostics(g.h)["gauss_resid_max"] == 0.0     # the reference: div E = 0
    P.pic_yee_update(g.h, P.PIC_E_FULL)
    P.pic_sync(g.h)
    E = [e.astype(np.float64) for e in g.get_fields()[0]]
    div = 0.0
    for a in range(dims):
        q = (np.roll(E[a], -1, 2 - a) - E[a]) / d[a]
        div = q if a == 0 else div + q
    assert np.abs(div).max() > 0.0
    assert P.pic_diagnostics(g.h)["gauss_resid_max"] == np.abs(div).max()
    g.close()
