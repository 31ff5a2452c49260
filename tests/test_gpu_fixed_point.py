"""FP64 tangent application with the fixed-point contraction (GPU tests): against
the atomic-free form, which contracts in FP64, on ragged grids, for inputs inside
the exponent range of the integer form and outside it (the point's warp then
contracts in FP64 too), with zero and with non-finite entries. Both forms round
each of a node's up to 8 x 15 x 15 products to 2^-53 of the row's largest, so they
agree within 1e-13 of the field's largest value."""
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


@pytest.mark.parametrize("shape", [(1, 1, 1), (5, 3, 3), (9, 7, 6), (12, 11, 10)])
def test_application_matches_the_fp64_contraction(binding, shape):
    nx, ny, nz = shape
    st = inputs.config_random(nx, ny, nz, seed=31, eta_lo=-0.03, eta_hi=0.3)
    P = binding.problem_from_state(st)
    P.linearize(abi.PFM_F64)
    v0 = np.random.default_rng(9).standard_normal(st.U.shape)
    part = v0.copy()
    part[:3] *= 1e-9  # displacements far below the order parameters
    wide = v0 * np.exp2(np.random.default_rng(2).integers(-60, 60, v0.shape))
    sparse = np.zeros_like(v0)
    sparse[4, v0.shape[1] // 2] = 1.0
    hole = v0.copy()
    hole[1, v0.shape[1] // 3] = np.nan
    hole[5, 0] = np.inf
    for name, v in (("plain", v0), ("small displacements", part), ("wide", wide), ("one entry", sparse),
                    ("zero", np.zeros_like(v0)), ("1e200", 1e200 * v0), ("1e-200", 1e-200 * v0), ("non-finite", hole)):
        vd = torch.from_numpy(v).cuda()
        P.set_deterministic(False)
        y = P.jacobian_apply(vd).cpu().numpy()
        P.set_deterministic(True)
        z = P.jacobian_apply(vd).cpu().numpy()
        assert (np.isfinite(y) == np.isfinite(z)).all(), name
        for f in range(y.shape[0]):
            ok = np.isfinite(z[f])
            scale = np.abs(z[f][ok]).max(initial=0.0)
            assert np.abs(y[f][ok] - z[f][ok]).max(initial=0.0) <= 1e-13 * scale, (name, f)
    P.close()
