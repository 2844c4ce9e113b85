"""Integer contractions on values of very different size inside one element
(dg_fixed.cuh, built for the host): every result is as close to the exact sum
as the FP64 chain is bound to be, (terms + 3) 2^-53 of the sum of the terms'
magnitudes."""
import numpy as np
import pytest

from fixed_host import fx, nodes, ptr  # noqa: F401

U = 2.0 ** -53
DEGREES = range(2, 8)
LD = np.longdouble


def along(a, l):
    """Axis of collapsed coordinate l last."""
    return np.moveaxis(a, 1 + l, -1)


@pytest.mark.parametrize("n", DEGREES)
def test_derivative_sum_keeps_line_scales(fx, n):  # noqa: F811
    rng = np.random.default_rng(n)
    D = nodes(n)[1]
    for dirs in range(1, 8):
        G = rng.uniform(-1, 1, (3, 5, n, n, n))
        for l in range(3):
            G[l] *= np.expand_dims(10.0 ** rng.uniform(-12, 0, (5, n, n)), 1 + l)
        G[:, 4] = 0.0
        out = np.empty((5, n, n, n))
        fx.t_dsum(n, ptr(G), dirs, ptr(out))
        ref, size = np.zeros(out.shape, LD), np.zeros(out.shape)
        for l in range(3):
            if dirs >> l & 1:
                g = along(G[l], l)[..., None]
                ref += np.moveaxis((g.astype(LD) * D).sum(-2), -1, 1 + l)
                size += np.moveaxis((np.abs(g) * np.abs(D).astype(float)).sum(-2), -1, 1 + l)
        assert (np.abs(out - ref) <= (n + 3) * U * size).all()
        assert (out[4] == 0).all()
