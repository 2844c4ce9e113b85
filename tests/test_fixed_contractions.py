"""Integer contractions on values of very different size inside one element
(dg_fixed.cuh, built for the host): every result is as close to the exact sum
as the FP64 chain is bound to be, (terms + 3) 2^-53 of the sum of the terms'
magnitudes."""
import numpy as np
import pytest

from fixed_host import fx, nodes, ptr, tables  # noqa: F401

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


def lifted(n, face, H, F, sign):
    """h = H + sign sum_f E_f^T F_f and the sum of its terms' magnitudes."""
    E = nodes(n)[2]
    h, size = H.astype(LD), np.abs(H)
    for l in range(3):
        for end in range(2):
            lf = face[2 * l + end]
            if lf < 0:
                continue
            shape = [1, 1, 1, 1]
            shape[1 + l] = n
            # face point x1 + n x2 of the two other coordinates
            term = sign * E[end].reshape(shape) * np.expand_dims(np.swapaxes(F[lf], 1, 2), 1 + l)
            h, size = h + term, size + np.abs(term).astype(float)
    return h, size


def spread(rng, n, nf):
    """Nodal values, and face values, of sizes from 1e-12 to 1: along a, and from node to node."""
    H = rng.uniform(-1, 1, (5, n, n, n)) * 10.0 ** rng.uniform(-12, 0, (5, n, n, n))
    F = rng.uniform(-1, 1, (nf, 5, n, n)) * 10.0 ** rng.uniform(-12, 0, (nf, 5, n, n))
    return H, F


@pytest.mark.parametrize("n", DEGREES)
@pytest.mark.parametrize("etype", range(4))
def test_lift_keeps_node_scales(fx, n, etype):  # noqa: F811
    rng = np.random.default_rng(10 * n + etype)
    face = tables(fx, n, etype)[1]
    H, F = spread(rng, n, face.max() + 1)
    for neg in (0, 1):
        out = np.empty_like(H)
        fx.t_lift(n, etype, ptr(H), ptr(F), neg, ptr(out))
        h, size = lifted(n, face, H, F, -1 if neg else 1)
        # besides the chain's nine roundings up to five units of 2^-57 of the largest value at the node, which
        # counts there with a coefficient of min |E| at least
        assert (np.abs(out - h) <= (9 + 5 / 16 / float(np.abs(nodes(n)[2]).min())) * U * size).all()


@pytest.mark.parametrize("n", DEGREES)
@pytest.mark.parametrize("etype", range(4))
def test_lift_to_modal_keeps_line_scales(fx, n, etype):  # noqa: F811
    rng = np.random.default_rng(10 * n + etype)
    V, face = tables(fx, n, etype)
    nf, nM = face.max() + 1, V.shape[1]
    H = rng.uniform(-1, 1, (5, n, n, n)) * 10.0 ** rng.uniform(-12, 0, (5, 1, n, n))
    F = rng.uniform(-1, 1, (nf, 5, n, n)) * 10.0 ** rng.uniform(-12, 0, (nf, 5, n, 1))
    for neg in (0, 1):
        h, size = lifted(n, face, H, F, -1 if neg else 1)
        ref = h.reshape(5, -1) @ V.astype(LD)
        # what meets on a line along a shares an exponent
        line = np.broadcast_to(size.max(axis=1, keepdims=True), size.shape)
        bound = (3 * n + 9) * U * (line.reshape(5, -1) @ np.abs(V))
        for stage in (0, 1):
            out = np.empty((5, nM))
            assert fx.t_lift_modal(n, etype, ptr(H), ptr(F), neg, stage, ptr(out)) == nM
            assert (np.abs(out - ref) <= bound).all()


@pytest.mark.parametrize("nM", [4, 18, 75])
def test_dense_product_keeps_small_modes(fx, nM):  # noqa: F811
    """A mildly bent element's inverse mass matrix on modes that decay over twelve orders."""
    rng = np.random.default_rng(nM)
    M = rng.uniform(-1, 1, (nM, nM)) * 1e-6
    M = np.diag(rng.uniform(0.5, 2, nM)) + M + M.T
    r = rng.uniform(-1, 1, (5, nM)) * 10.0 ** np.linspace(0, -12, nM)
    out = np.empty((5, nM))
    fx.t_dense(nM, ptr(M), ptr(r), ptr(out))
    ref = r.astype(LD) @ M.astype(LD)
    assert (np.abs(out - ref) <= (nM + 3) * U * (np.abs(r) @ np.abs(M))).all()


def kinds(a):
    """0 finite, 1 +infinity, 2 -infinity, 3 NaN"""
    return np.where(np.isnan(a), 3, np.where(np.isposinf(a), 1, np.where(np.isneginf(a), 2, 0)))


@pytest.mark.parametrize("n", DEGREES)
@pytest.mark.parametrize("etype", range(4))
@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan, 1e303, 3e-310])
def test_extreme_values(fx, n, etype, value):  # noqa: F811
    """One infinity, NaN or huge value, or a variable of subnormals.  The one-shot maps give the FP64 sums:
    infinities by value, gradual underflow.  The phases of a residual are not finite exactly where the FP64 sums
    are not (NaN there), and lose what lies below the normal range."""
    rng = np.random.default_rng(100 * n + etype)
    V, face = tables(fx, n, etype)
    D, E = (m.astype(float) for m in nodes(n)[1:])
    nf, nM = face.max() + 1, V.shape[1]

    def field(*shape):
        a = rng.uniform(-1, 1, shape)
        if value == 3e-310:
            a[0] *= value
        else:
            a[0].flat[rng.integers(a[0].size)] = value
        return a

    def check(got, terms, ieee=False):
        """terms: the products to be summed, along the last axis"""
        size = np.abs(np.where(np.isfinite(terms), terms, 0)).sum(-1)
        ref = terms.sum(-1)
        if ieee:
            assert (kinds(got) == kinds(ref)).all()
        else:
            assert (np.isnan(got) == ~np.isfinite(ref)).all() and not np.isinf(got).any()
        ok = np.isfinite(ref)
        if value == 1e303 and not ieee:
            return            # the accuracy beside a large value: the tests above
        # chains of three passes; 400 last bits of subnormals, or the end of the normal range
        tiny = 400 * 2.0 ** -1074 if ieee else 2.0 ** -1022
        assert (np.abs(got - ref)[ok] <= (6 * n + 20) * U * size[ok] + tiny).all()

    with np.errstate(all="ignore"):
        Q, W = field(5, nM), field(5, n, n, n)
        A, R, tr = np.empty((5, n ** 3)), np.empty((5, nM)), np.empty((nf, 5, n, n))
        for ieee in (0, 1):
            fx.t_nodal(n, etype, ieee, ptr(Q), ptr(A), ptr(tr))
            check(A, Q[:, None, :] * V[None], ieee)
            fx.t_modal(n, etype, ieee, ptr(W), ptr(R))
            check(R, W.reshape(5, -1)[:, None, :] * V.T[None], ieee)
        g = np.empty((3, 5, n, n, n))
        fx.t_grad(n, ptr(W), ptr(g))
        for l in range(3):
            check(along(g[l], l), along(W, l)[..., None, :] * D)
        G = rng.uniform(-1, 1, (3, 5, n, n, n))
        G[int(rng.integers(3))] = W
        out = np.empty((5, n, n, n))
        fx.t_dsum(n, ptr(G), 7, ptr(out))
        check(out, np.concatenate([np.moveaxis(along(G[l], l)[..., None, :] * D.T, -2, 1 + l) for l in range(3)], axis=-1))
        # the lift, of an extreme node or an extreme face value
        for H, F in ((W, rng.uniform(-1, 1, (nf, 5, n, n))), (rng.uniform(-1, 1, W.shape), field(5, nf, n, n).swapaxes(0, 1).copy())):
            if value == 3e-310:
                H, F = H * 1.0, F * 1.0
                H[0] = rng.uniform(-1, 1, H[0].shape) * value
                F[:, 0] = rng.uniform(-1, 1, F[:, 0].shape) * value
            terms = [H]
            for k in range(6):
                if face[k] >= 0:
                    shape = [1, 1, 1, 1]
                    shape[1 + k // 2] = n
                    f = np.expand_dims(np.swapaxes(F[face[k]], 1, 2), 1 + k // 2)
                    terms.append(np.broadcast_to(-E[k % 2].reshape(shape) * f, H.shape))
            terms = np.stack(terms, axis=-1)
            fx.t_lift(n, etype, ptr(H), ptr(F), 1, ptr(out))
            check(out, terms)
            both = (terms.reshape(5, 1, n ** 3, -1) * V.T[None, :, :, None]).reshape(5, nM, -1)
            for stage in (0, 1):
                fx.t_lift_modal(n, etype, ptr(H), ptr(F), 1, stage, ptr(R))
                check(R, both)


@pytest.mark.parametrize("n", [3, 5, 6])
def test_derivative_sum_does_not_lean(fx, n):  # noqa: F811
    """The mean error of many results, of lines on different exponents, is a small part of a single one's: errors that
    lean one way add up in the integral behind (about 2 units of 2^-53 each at n = 6; 0.1 is five deviations of the mean)."""
    rng = np.random.default_rng(n)
    D = nodes(n)[1]
    err = []
    for _ in range(60):
        G = rng.uniform(0.3, 1, (3, 5, n, n, n)) * 2.0 ** rng.uniform(-4, 0, (3, 5, 1, 1, 1)) * rng.choice([-1, 1], (3, 5, 1, 1, 1))
        out, ref = np.empty((5, n, n, n)), np.zeros((5, n, n, n), LD)
        fx.t_dsum(n, ptr(G), 7, ptr(out))
        for l in range(3):
            ref += np.moveaxis((along(G[l], l)[..., None].astype(LD) * D).sum(-2), -1, 1 + l)
        err.append(out - ref)
    assert abs(np.concatenate(err).mean()) < 0.1 * U
