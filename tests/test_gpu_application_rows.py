"""Rounding of the FP64 tangent application row by row (GPU test): every entry of
J v is within 64 units of 2^-53 of (|J| |v|) at its own node and field, also where the
penalty on one order parameter is far above every other entry of the Hessian. The
bound counts the roundings on a path from v to y: at most 9 in the gather to the Gauss
points, 16 in the contraction with the stored Hessian, 2 in its weight, 9 in the
scatter and 8 in the sum over a node's elements, 44 in all. The reference takes the
stored Hessians as they are, in extended precision; the interface energy is switched
off so that the rows consist of the contraction alone."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2011_08802_gb300 import abi, inputs  # noqa: E402

pytestmark = pytest.mark.gpu

LD = np.longdouble


@pytest.fixture(scope="module")
def binding():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2011_08802_gb300 import binding as b
    return b


def _point_operator(h):
    """z = (grad u, eta) at the 8 Gauss points from the 9 x 8 nodal values of one element."""
    ga = (LD(1) - 1 / np.sqrt(LD(3))) / 2
    B = np.zeros((8, 15, 9, 8), dtype=LD)
    for q in range(8):
        xi = [1 - ga if (q >> d) & 1 else ga for d in range(3)]
        for a in range(8):
            phi = [xi[d] if (a >> d) & 1 else 1 - xi[d] for d in range(3)]
            dphi = [(LD(1) if (a >> d) & 1 else LD(-1)) / h[d] for d in range(3)]
            for J in range(3):
                g = dphi[J]
                for d in range(3):
                    g = g * (phi[d] if d != J else 1)
                for i in range(3):
                    B[q, 3 * i + J, i, a] = g
            for k in range(6):
                B[q, 9 + k, 3 + k, a] = phi[0] * phi[1] * phi[2]
    return B


@pytest.mark.parametrize("eps_eta", [1e3, 1e6, 1e9])
@pytest.mark.parametrize("part", ["all", "displacements", "order parameters", "one order parameter"])
def test_every_row_rounds_like_its_own_sum(binding, eps_eta, part):
    nx, ny, nz = 3, 2, 2
    st = inputs.config_random(nx, ny, nz, seed=12, eta_lo=-0.03, eta_hi=0.3, Lx=3.0, Ly=2.0, Lz=2.0)
    prm = abi.params_from_material(st.material, st.tau, gamma_scale=0.0)
    prm.eps_eta = eps_eta
    P = binding.problem_from_state(st, params=prm)
    P.linearize(abi.PFM_F64)
    v = np.random.default_rng(3).standard_normal(st.U.shape)
    if part == "displacements":
        v[3:] = 0.0
    elif part == "order parameters":
        v[:3] = 0.0
    elif part == "one order parameter":
        v[:4] = v[5:] = 0.0
    y = P.jacobian_apply(torch.from_numpy(v).cuda()).cpu().numpy()
    ne = nx * ny * nz
    packed = P.get_hessians(0, ne)
    P.close()
    H = np.zeros((ne, 8, 15, 15))
    iu = np.triu_indices(15)
    H[:, :, iu[0], iu[1]] = packed
    H[:, :, iu[1], iu[0]] = packed
    assert (np.abs(H[:, :, 9:, 9:]).max((2, 3)) > 0.5 * eps_eta).any()  # the penalty is active
    h = st.mesh.h
    B = _point_operator(h)
    w = LD(h[0]) * LD(h[1]) * LD(h[2]) / 8
    mask = st.mask.astype(bool)
    vf = np.where(mask, 0.0, v).astype(LD)
    ref, mag = np.zeros(v.shape, dtype=LD), np.zeros(v.shape, dtype=LD)
    for e in range(ne):
        ei, ej, ek = e % nx, (e // nx) % ny, e // (nx * ny)
        nodes = [(ei + (a & 1)) + (nx + 1) * ((ej + (a >> 1 & 1)) + (ny + 1) * (ek + (a >> 2))) for a in range(8)]
        x = vf[:, nodes]
        for q in range(8):
            Hq = H[e, q].astype(LD)
            ref[:, nodes] += w * np.einsum("zfa,z->fa", B[q], Hq @ np.einsum("zfa,fa->z", B[q], x))
            mag[:, nodes] += w * np.einsum("zfa,z->fa", np.abs(B[q]),
                                           np.abs(Hq) @ np.einsum("zfa,fa->z", np.abs(B[q]), np.abs(x)))
    ref, mag = np.where(mask, v, ref), np.where(mask, 0, mag)
    err = np.abs(y - ref)
    assert (err <= 64 * LD(2) ** -53 * mag).all(), float((err / np.where(mag > 0, mag, 1)).max() * 2.0 ** 53)
