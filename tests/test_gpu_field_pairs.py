"""The one-pass end of a step (by pairs of steps of one call, through the unused
particle pool) against the two passes in place, to the last bit: uncharged particles
make the pool and add no current, so the fields do not depend on any order of
sums.  Odd sizes down to the smallest grid, both precisions, an antenna next to and
away from its plane's neighbours, the vector potential, and a batch of unequal runs;
the number of launches shows that the one pass was taken."""
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


def particles(rng, n, dims):
    count = 3 * n[0] * n[1] * n[2]
    x = np.zeros((3, count))
    for a in range(dims):
        x[a] = rng.uniform(0.0, n[a], count)
    return x, rng.normal(0.0, 1.0, (3, count))


def launches(P, h, k):
    before = P.pic_kernel_launches(h)
    P.pic_step(h, k)
    return P.pic_kernel_launches(h) - before


def by_parts(P, h):
    P.pic_yee_update(h, P.PIC_B_HALF)
    P.pic_gather_push(h)
    P.pic_deposit_current(h)
    P.pic_yee_update(h, P.PIC_B_HALF)
    P.pic_yee_update(h, P.PIC_E_FULL)


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("dims,n", [(2, (11, 13, 1)), (2, (64, 9, 1)), (3, (9, 11, 10)), (3, (33, 10, 12))])
@pytest.mark.parametrize("extra", ["none", "antenna 1", "antenna 4", "antenna 8", "vector potential"])
def test_one_pass_is_the_two_passes(P, prec, dims, n, extra):
    rng = np.random.Generator(np.random.PCG64(n[0] + 89))
    x, w = particles(rng, n, dims)
    fields = None
    want = None
    for split in ([1] * 7, [7], [2, 5], [6, 1], "parts"):
        g = P.Grid(P.make_desc(dims, n, (1.0,) * 3, 0.04, 10.0, prec, tile=(4, 4, 4), halo=0, sort_interval=1000))
        if fields is None:
            fields = [[rng.normal(size=g.shape) for _ in range(3)] for _ in range(3)]
        g.set_fields(fields[0], fields[1])
        g.load(0, 0.0, 1.0, 1.0, x, w)
        if extra.startswith("antenna"):
            plane = int(extra.split()[1])
            P.pic_set_antenna(g.h, 0, 1 + plane % 2, plane, 0.5, 1.3, 2.0, 7)
        if extra == "vector potential":
            P.pic_set_vector_potential(g.h, [a.astype(g.dtype) for a in fields[2]], set_B=False)
        if split == "parts":
            for _ in range(7):
                by_parts(P, g.h)
        else:
            took = [launches(P, g.h, k) for k in split]
            if split == [1] * 7:
                one = took[-1]
            else:
                assert took == [k * one - (k - k % 2) for k in split]   # a launch less in each step of a pair
        P.pic_sync(g.h)
        E, B, J = g.get_fields()
        got = E + B
        if extra == "vector potential":
            A = [np.empty_like(E[0]) for _ in range(3)]
            P.pic_get_vector_potential(g.h, A)
            got += A
        assert not any(j.any() for j in J)
        if want is None:
            want = got
        for u, v in zip(got, want):
            np.testing.assert_array_equal(u, v)
        g.close()


@pytest.mark.parametrize("prec", [0, 1])
def test_a_batch_of_unequal_runs(P, prec):
    sizes = [(31, 24, 1), (24, 40, 1), (57, 25, 1)]
    rng = np.random.Generator(np.random.PCG64(90))
    parts = [particles(rng, n, 2) for n in sizes]
    fields = [[[rng.normal(size=(1, n[1], n[0])) for _ in range(3)] for _ in range(2)] for n in sizes]
    got = []
    for split in ([1] * 6, [6], [3, 3], [5, 1]):
        b = P.Batch([P.make_desc(2, n, (1.0,) * 3, 0.04, 10.0, prec, tile=(8, 8, 1), sort_interval=3) for n in sizes])
        dt = np.float64 if prec == 0 else np.float32
        for r, (x, w) in enumerate(parts):
            P.pic_set_fields_run(b.h, r, *[[np.ascontiguousarray(f, dtype=dt) for f in fs] for fs in fields[r]])
            b.load_run(r, 0, 0.0, 1.0, 1.0, x, w)
        for k in split:
            P.pic_step(b.h, k)
        P.pic_sync(b.h)
        got.append([f for r in range(len(sizes)) for fs in b.get_fields_run(r)[:2] for f in fs])
        b.close()
    for other in got[1:]:
        for u, v in zip(other, got[0]):
            np.testing.assert_array_equal(u, v)
