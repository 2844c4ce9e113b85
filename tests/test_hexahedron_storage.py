"""A hexahedron's storage (scaled nodal values) and back: the modal state
returns to rounding, so a step carries no error of the tables into the state."""
import numpy as np
import pytest

from fixed_host import fx, ptr  # noqa: F401


@pytest.mark.parametrize("n", range(2, 8))
def test_state_returns(fx, n):  # noqa: F811
    rng = np.random.default_rng(n)
    nM = n ** 3
    Q = rng.uniform(-1, 1, (5, nM)) * 10.0 ** rng.uniform(-6, -1, (5, nM))
    Q[:, 0] = [1.2, -0.3, 0.2, 0.1, 180.0]
    out = np.empty_like(Q)
    assert fx.t_storage(n, ptr(Q), ptr(out)) == nM
    # a node's value, its scaled value, the factor of the way back and the scaled product are rounded once each
    # (half a unit), the result once: relative to the constant mode, which every node carries
    big = np.abs(Q[:, 0])
    assert (np.abs(out[:, 0] - Q[:, 0]) <= 2.6 * 2.0 ** -53 * 1.2 * big).all()
    # the other modes take those roundings through the orthogonal transform
    assert (np.abs(out - Q).max(axis=1) <= 2.6 * 2.0 ** -53 * 1.2 * np.sqrt(nM) * big).all()
