"""The blocked Gauss-Jordan inverse of the dense coarse operator (GPU tests).
On a one-level hierarchy the V-cycle is the coarse solve alone, so z = M r is
K^-1 r; K is read out with FP64 tangent applications to unit vectors and
inverted by LAPACK. Orders around the panel width (16), the tile (32) and the
cluster splits (128 rows per CTA up to the 8-CTA cluster). Bound: the forward
error of Gauss-Jordan elimination with partial pivoting, a modest multiple of
n u cond_1(K) (Higham, Accuracy and Stability of Numerical Algorithms, Ch. 14)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2011_08802_gb300 import abi, inputs  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def binding():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2011_08802_gb300 import binding
    return binding


# 9 (nx+1)(ny+1)(nz+1) unknowns: 72, 108, 162, 243, 432, 1125, 4032
@pytest.mark.parametrize("shape", [(1, 1, 1), (2, 1, 1), (2, 2, 1), (2, 2, 2), (3, 3, 2), (4, 4, 4), (7, 6, 7)])
@pytest.mark.parametrize("n_var", [6, 12])
def test_one_level_vcycle_is_the_inverse(binding, shape, n_var):
    if n_var == 12 and shape[0] > 4:
        pytest.skip("more unknowns than the coarsest level may have")
    st = inputs.config_random(*shape, seed=3, eta_lo=0.0, eta_hi=0.3 if n_var == 6 else 0.15, Lx=8.0, Ly=8.0, Lz=8.0,
                              top=False, n_var=n_var)
    P = binding.problem_from_state(st, n_levels=1)
    P.linearize(abi.PFM_F64)
    n = P.shape[0] * P.shape[1]
    K = np.empty((n, n))
    e = torch.zeros(n, dtype=torch.float64, device="cuda")
    for c in range(n):
        e[c] = 1.0
        K[:, c] = P.jacobian_apply(e.reshape(P.shape)).cpu().numpy().reshape(-1)
        e[c] = 0.0
    X = np.linalg.inv(K)
    cond = np.linalg.norm(K, 1) * np.linalg.norm(X, 1)
    r = np.random.default_rng(1).standard_normal(n)
    z = P.vcycle(torch.from_numpy(r).cuda().reshape(P.shape)).cpu().numpy().reshape(-1)
    ref = np.linalg.solve(K, r)
    assert np.linalg.norm(z - ref) <= 8 * n * np.finfo(float).eps * cond * np.linalg.norm(ref)
    assert np.linalg.norm(K @ z - r) <= 8 * n * np.finfo(float).eps * cond * np.linalg.norm(r)
    P.close()


def test_singular_operator_is_reported(binding):
    """No stiffness, no interface energy, no dissipation: a zero operator."""
    st = inputs.config_random(2, 2, 2, seed=3, top=False)
    c = dict(st.material, C11=0.0, C12=0.0, C44=0.0, gamma_am=0.0, gamma_mm=0.0, eps_eta=0.0, mobility=float("inf"))
    P = binding.problem_from_state(st, n_levels=1, params=abi.params_from_material(c, st.tau))
    with pytest.raises(binding.PfmError) as err:
        P.linearize(abi.PFM_F64)
    assert err.value.status == 6
    P.close()
