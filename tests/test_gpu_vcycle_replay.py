"""V-cycles after the first one of a linearisation (GPU test): they replay a CUDA
graph, and have to give what a fresh handle's first V-cycle, issued launch by launch,
gives. In the atomic-free mode both are the same operations in the same order, so they
are compared bitwise: repeated calls, other inputs and output buffers, changed smoother
options and back, the binary16 store switched on and off, a new state, another stream.
With atomics the sums differ in their order only."""
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


def _state(shape, seed):
    return inputs.config_random(*shape, seed=seed, eta_lo=-0.02, eta_hi=0.3)


def _fresh(binding, st, prec, r, opts, half=False, det=True):
    P = binding.problem_from_state(st)
    P.set_deterministic(det)
    P.set_preconditioner_store(half)
    P.linearize(prec)
    z = P.vcycle(r, opts=opts)
    P.close()
    return z


@pytest.mark.parametrize("shape", [(8, 8, 8), (9, 7, 6)])  # nested and non-nested levels
@pytest.mark.parametrize("prec, dtype", [(abi.PFM_F32, torch.float32), (abi.PFM_F64, torch.float64)])
def test_replayed_vcycles_equal_direct_ones(binding, shape, prec, dtype):
    st, st2 = _state(shape, 5), _state(shape, 6)
    gen = torch.Generator("cuda").manual_seed(4)
    rs = [torch.randn(st.U.shape, generator=gen, device="cuda", dtype=dtype) for _ in range(3)]
    a = abi.default_opts(prec)
    b = abi.default_opts(prec, nu_pre=3, nu_post=2, cheb_lo=0.1)
    ref = {(i, o): _fresh(binding, st, prec, rs[i], opt) for i in range(3) for o, opt in (("a", a), ("b", b))}
    P = binding.problem_from_state(st)
    P.set_deterministic(True)
    P.linearize(prec)
    for i, o in [(0, "a"), (0, "a"), (1, "a"), (2, "a"), (1, "b"), (1, "b"), (2, "a"), (2, "b"), (0, "a")]:
        z = P.vcycle(rs[i], opts=a if o == "a" else b)
        assert torch.equal(z, ref[i, o]), (i, o)
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    P.set_stream(s)
    z = P.vcycle(rs[1], opts=a)
    s.synchronize()
    assert torch.equal(z, ref[1, "a"])
    P.set_stream(torch.cuda.current_stream())
    # another state: new coefficients and stores behind the same graph
    P.set_state(torch.from_numpy(st2.U).cuda(), torch.from_numpy(st2.Un).cuda())
    P.linearize(prec)
    new = _fresh(binding, st2, prec, rs[0], a)
    for _ in range(3):
        assert torch.equal(P.vcycle(rs[0], opts=a), new)
    if prec == abi.PFM_F32:
        for half in (True, False):
            P.set_preconditioner_store(half)
            P.linearize(prec)
            want = _fresh(binding, st2, prec, rs[2], a, half)
            for _ in range(3):
                assert torch.equal(P.vcycle(rs[2], opts=a), want)
    # the atomic-free switch between two V-cycles of one linearisation
    P.set_deterministic(False)
    got = [P.vcycle(rs[1], opts=a) for _ in range(3)]
    P.set_deterministic(True)
    want = P.vcycle(rs[1], opts=a)
    assert torch.equal(want, _fresh(binding, st2, prec, rs[1], a))
    tol = 1e-4 if prec == abi.PFM_F32 else 1e-12
    for z in got:
        assert torch.linalg.norm(z - want) <= tol * torch.linalg.norm(want)
    P.close()
