"""Units scaled by a power of two (GPU test): energies, stiffnesses and rate constants
times 2^k leave the kinematics alone and scale residual, Hessians and operators by 2^k
exactly, up to the rounding of the forms that the kernels choose by exponent. At
k = 0 the order-parameter columns of the Hessian and the coarse inverse's updates are
formed in fixed point, at k = +-600 they are outside its range of exponents and take
their FP64 sums, at k = +-200 they are near its ends."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2011_08802_gb300 import abi, inputs  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def binding():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2011_08802_gb300 import binding as b
    return b


def _scaled(st, k):
    p = abi.params_from_material(st.material, st.tau)
    s = 2.0 ** k
    for i in range(7):
        for j in range(36):
            p.Lvoigt[i][j] *= s
        p.F0[i] *= s
        p.mobility[i] /= s
    p.gamma_scale *= s
    p.eps_eta *= s
    return p


@pytest.mark.parametrize("k", [-600, -200, 200, 600])
def test_scaled_units_give_scaled_results(binding, k):
    """Hessians: both forms are within 1e-12 of the largest entry (tests of the point
    physics). Coarse inverse, on one level: Gauss-Jordan with partial pivoting, error
    8 n 2^-53 cond(K) as in the test of the coarse inverse."""
    st = inputs.config_random(3, 2, 2, seed=9, eta_lo=-0.02, eta_hi=0.3)
    s = 2.0 ** -k
    r = torch.from_numpy(np.random.default_rng(1).standard_normal(st.U.shape)).cuda()
    r[torch.from_numpy(st.mask).cuda().bool()] = 0.0
    got = []
    for p in (abi.params_from_material(st.material, st.tau), _scaled(st, k)):
        P = binding.problem_from_state(st, n_levels=1, params=p)
        f = 1.0 if not got else s
        R, e = P.residual(energy=True)
        P.linearize(abi.PFM_F64)
        H = P.get_hessians(0, P.n_elems)
        z = P.vcycle(r, opts=abi.default_opts(abi.PFM_F64))
        got.append((R.cpu().numpy() * f, e * f, H * f, z.cpu().numpy().reshape(-1) / f))
        P.close()
    (R0, e0, H0, z0), (R1, e1, H1, z1) = got
    assert np.abs(R1 - R0).max() <= 1e-13 * np.abs(R0).max()
    assert abs(e1 - e0) <= 1e-12 * abs(e0)
    assert np.abs(H1 - H0).max() <= 1e-12 * np.abs(H0).max()
    n = z0.size
    P = binding.problem_from_state(st, n_levels=1)
    P.linearize(abi.PFM_F64)
    K = np.empty((n, n))
    for i in range(n):
        v = torch.zeros(n, dtype=torch.float64, device="cuda")
        v[i] = 1.0
        K[:, i] = P.jacobian_apply(v.reshape(r.shape)).cpu().numpy().reshape(-1)
    P.close()
    free = ~st.mask.reshape(-1).astype(bool)
    K, b = K[np.ix_(free, free)], r.cpu().numpy().reshape(-1)[free]
    ref = np.linalg.solve(K, b)
    tol = 8 * n * 2.0 ** -53 * np.linalg.cond(K) * np.linalg.norm(ref)
    for z in (z0, z1):
        assert not z[~free].any()
        assert np.linalg.norm(z[free] - ref) <= tol
