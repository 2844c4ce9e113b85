"""Infinities through the one-shot maps, whose results are the caller's: by
value, as in plain FP64 sums, in the element that holds them and nowhere
else; the phases of a residual keep no finite value that depends on one."""
import numpy as np
import pytest

from gpu_util import make_box

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [1, 4, 6])
@pytest.mark.parametrize("value", [np.inf, -np.inf])
def test_infinite_mean_of_an_element(N, value):
    import paper_2511_08020_gb300 as dg
    box = make_box("four", 4)
    mesh = dg.Mesh(box, N)
    rng = np.random.default_rng(N)
    nQ = (N + 1) ** 3
    vals = rng.uniform(0.5, 1, (box.n_elems, 5, nQ))
    vals[:, 4] += 50.0
    Q = mesh.get_state(mesh.project(torch.from_numpy(vals).cuda()))
    Q = torch.as_tensor(Q).double().cpu().numpy().copy()
    nM = [(N + 1) ** 3, (N + 1) ** 2 * (N + 2) // 2, (N + 1) * (N + 2) * (2 * N + 3) // 6, (N + 1) * (N + 2) * (N + 3) // 6]
    off = np.concatenate([[0], np.cumsum([5 * nM[t] for t in box.etype])])
    bad = [int(np.nonzero(box.etype == t)[0][0]) for t in range(4)]     # one element of each type
    clean = mesh.eval_nodal(mesh.set_state(torch.from_numpy(Q).cuda()))
    clean = torch.as_tensor(clean).cpu().numpy().reshape(box.n_elems, 5, nQ)
    for e in bad:
        Q[off[e] + 4 * nM[box.etype[e]]] = value                        # the constant mode of the energy
    Qs = mesh.set_state(torch.from_numpy(Q).cuda())
    got = torch.as_tensor(mesh.eval_nodal(Qs)).cpu().numpy().reshape(box.n_elems, 5, nQ)
    for e in range(box.n_elems):
        if e in bad:
            assert (got[e, 4] == value).all()
            np.testing.assert_allclose(got[e, :4], clean[e, :4], rtol=0, atol=1e-13)
        else:
            np.testing.assert_array_equal(got[e], clean[e])
    back = torch.as_tensor(mesh.get_state(Qs)).cpu().numpy()
    for e in bad:
        assert back[off[e] + 4 * nM[box.etype[e]]] == value
    # point values: the projection's constant mode is infinite, not NaN
    vals[bad[0], 4, nQ // 2] = value
    P = torch.as_tensor(mesh.get_state(mesh.project(torch.from_numpy(vals).cuda()))).cpu().numpy()
    assert P[off[bad[0]] + 4 * nM[0]] == value
    R = torch.as_tensor(mesh.get_state(mesh.rhs(Qs))).cpu().numpy()
    for e in bad:
        assert not np.isfinite(R[off[e] + 4 * nM[box.etype[e]]:off[e + 1]]).any()
    far = [e for e in range(box.n_elems) if np.isfinite(R[off[e]:off[e + 1]]).all()]
    assert far
