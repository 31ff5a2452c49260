"""The nodal form of the gradient energy (GPU tests). Residual and tangent are
affine in gamma_scale, so the difference of two values of it isolates the
interface energy: on the order-parameter rows its residual is
sum_l (G_kl A + C_kl M) eta_l + c_0k M 1, with the stiffness A and mass matrix M of
trilinear elements (tensor products of their 1-D matrices) and the condensed
coefficients of Eq. IntEnergy. Grids at the edges of the kernel's chunks of four
node planes, one element wide, and ragged. Bound: rounding of the two values
that are subtracted, 64 units of the arithmetic's last place."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
sparse = pytest.importorskip("scipy.sparse")

from paper_2011_08802_gb300 import abi, inputs  # noqa: E402

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1, 1), (1, 1, 6), (3, 2, 3), (2, 5, 4), (7, 1, 7), (33, 2, 8)]


@pytest.fixture(scope="module")
def binding():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2011_08802_gb300 import binding
    return binding


def _matrices(mesh):
    """A (gradient) and M (value) on the node grid, x fastest."""
    K1, M1 = [], []
    for n, h in zip((mesh.nx, mesh.ny, mesh.nz), mesh.h):
        K, M = sparse.lil_matrix((n + 1, n + 1)), sparse.lil_matrix((n + 1, n + 1))
        for e in range(n):
            K[e:e + 2, e:e + 2] += np.array([[1, -1], [-1, 1]]) / h
            M[e:e + 2, e:e + 2] += np.array([[2, 1], [1, 2]]) * h / 6
        K1.append(K.tocsr())
        M1.append(M.tocsr())

    def kron(x, y, z):
        return sparse.kron(z, sparse.kron(y, x)).tocsr()

    A = kron(K1[0], M1[1], M1[2]) + kron(M1[0], K1[1], M1[2]) + kron(M1[0], M1[1], K1[2])
    return A, kron(*M1)


def _coefficients(prm, nv):
    n = nv + 1
    c = np.array([[0.0 if i == j else 4 * prm.gamma[i][j] / (math.pi * prm.ell[i][j]) for j in range(n)]
                  for i in range(n)])
    ell2 = np.array([[prm.ell[i][j] ** 2 for j in range(n)] for i in range(n)])
    T = np.vstack([-np.ones((1, nv)), np.eye(nv)])
    return T.T @ (-c * ell2) @ T, T.T @ c @ T, c[0, 1:]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("n_var", [6, 12])
@pytest.mark.parametrize("det", [False, True])
def test_interface_energy_is_the_nodal_operator(binding, shape, n_var, det):
    st = inputs.config_random(*shape, seed=7, eta_lo=0.0, eta_hi=0.3 if n_var == 6 else 0.15, Lx=9.0, Ly=7.0, Lz=8.0,
                              top=False, n_var=n_var)
    A, M = _matrices(st.mesh)
    v = torch.from_numpy(inputs.direction_vectors(st, 1, seed=1)[0]).cuda()
    vf = v.to(torch.float32)
    got = []
    for s in (1.0, 2.0):
        prm = abi.params_from_material(st.material, st.tau, gamma_scale=s)
        P = binding.problem_from_state(st, params=prm)
        P.set_deterministic(det)
        R, e = P.residual(energy=True)
        P.linearize(abi.PFM_F32)
        got.append([x.cpu().numpy() for x in (R, P.jacobian_apply(v), P.jacobian_apply_mixed(vf))] + [e])
        P.close()
    G, Cc, c0 = _coefficients(abi.params_from_material(st.material, st.tau), n_var)
    eta = st.U[3:]
    one = np.ones(st.mesh.n_nodes)

    def op(x):  # rows of (G A + C M) x
        return G @ (A @ x.T).T + Cc @ (M @ x.T).T

    refs = [op(eta) + np.outer(c0, M @ one), op(v[3:].cpu().numpy()), op(vf[3:].double().cpu().numpy())]
    for k, (ref, eps) in enumerate(zip(refs, (2.0 ** -52, 2.0 ** -52, 2.0 ** -46))):
        d = got[1][k][3:] - got[0][k][3:]
        assert np.abs(d - ref).max() <= 64 * eps * np.abs(got[1][k]).max(), (k, np.abs(d - ref).max())
    e_ref = 0.5 * np.sum(eta * op(eta)) + np.sum(c0[:, None] * eta * (M @ one))
    assert abs((got[1][3] - got[0][3]) - e_ref) <= 64 * 2.0 ** -52 * (abs(got[1][3]) + abs(got[0][3])) + \
        1e-13 * np.abs(eta * op(eta)).sum()
