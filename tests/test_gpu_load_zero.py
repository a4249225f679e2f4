"""Positions at the ends of the box: a position of -0.0 is cell 0 with offset +0.0,
bit for bit, and N wraps to 0, in both precisions and for every load path."""
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
@pytest.mark.parametrize("dims,order2", [(2, 3), (3, 3), (3, 5)])
def test_ends_of_the_box(P, prec, dims, order2):
    n = (16, 18, 1) if dims == 2 else (16, 18, 20)
    ends = [-0.0, 0.0, "N", "-N", 0.5, "below N"]
    x = np.zeros((3, len(ends)))
    for a in range(dims):
        N = float(n[a])
        x[a] = [{"N": N, "-N": -N, "below N": N - 0.25}.get(e, e) for e in ends]
    g = P.Grid(P.make_desc(dims, n, (1.0,) * 3, 0.02, 20.0, prec, tile=(4, 4, 4), order2=order2))
    g.load(0, -1.0, 1.0, 1.0, x, np.zeros_like(x))
    cell, off, _, ident = g.particles(0)
    order = np.argsort(ident)
    want = np.array([0.0, 0.0, 0.0, 0.0, 0.5, 0.75])
    for a in range(dims):
        got = off[a][order]
        np.testing.assert_array_equal(got, want)
        assert not np.signbit(got).any()
    last = n[0] - 1 + n[0] * (n[1] - 1 + (n[1] * (n[2] - 1) if dims == 3 else 0))
    np.testing.assert_array_equal(cell[order], [0, 0, 0, 0, 0, last])
    g.close()
