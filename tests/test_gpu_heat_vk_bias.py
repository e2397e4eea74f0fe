"""Rounding of the variable-coefficient step has no bias, on grids whose axes have
spacings of their own (weighted axis sums) as on cubes: the mean error over all
points against extended precision stays within what unbiased rounding leaves."""
import numpy as np
import pytest

from tests.gpu_util import lib, require_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(150, 170, 160), (160, 160, 160)])
def test_mean_error(shape):
    require_cuda()
    pkg = lib()
    L, steps, r = np.longdouble, 2, 1.0 / (12 * 0.95)
    if np.finfo(L).nmant <= 52:
        pytest.skip("no extended precision")
    nodes = [np.arange(n + 2).astype(L) / L(n + 1) for n in shape]
    pi = L("3.14159265358979323846264338327950288")
    s, c = [np.sin(pi * v) for v in nodes], [np.cos(pi * v) for v in nodes]

    def outer(v):
        return v[0][:, None, None] * v[1][None, :, None] * v[2][None, None, :]

    rng = np.random.default_rng(7)
    u0 = outer([v[1:-1] for v in s]).astype(np.float64) + 0.01 * rng.uniform(-1, 1, size=shape)
    with pkg.Heat(*shape[::-1], r, flags=pkg.HS_VARKAPPA) as h:
        got = h.upload(u0).step(steps).read()
    # the same coefficients, rounded to FP64 as the library keeps them
    dt = r * min(1.0 / (n + 1) for n in shape) ** 2
    kap = (L("0.5") + L("0.45") * outer(s)).astype(np.float64).astype(L)
    fdt = (L(dt) * (1 + outer(c))).astype(np.float64).astype(L)[1:-1, 1:-1, 1:-1]
    beta = [L(dt) * L(n + 1) ** 2 / 2 for n in shape]
    inner = (slice(1, -1),) * 3
    faces = [(d, tuple(sl if a == d else slice(1, -1) for a in range(3)))
             for d in range(3) for sl in (slice(0, -2), slice(2, None))]
    weight = [beta[d] * (kap[inner] + kap[f]) for d, f in faces]
    u = np.zeros(kap.shape, dtype=L)
    u[inner] = u0
    for _ in range(steps):
        c0 = u[inner]
        new = c0 + fdt
        for (_, f), w in zip(faces, weight):
            new = new + w * (u[f] - c0)
        u[inner] = new
    err = got.astype(L) - u[inner]
    scale = np.abs(u).max()
    # a step rounds each value twice (u + dt f, and the sum), each time to within
    # 2^-54 of the largest: a standard deviation of 2^-54 / sqrt(3), independent from
    # point to point but not from step to step (the same dt f is added again).  Six
    # standard deviations of the mean; three products rounded down left 3e-19 a step.
    bound = 6 * steps * np.sqrt(2.0 / 3.0) * 2.0 ** -54 / np.sqrt(u0.size)
    assert abs(err.mean()) <= bound * scale, (float(err.mean() / scale), bound)
