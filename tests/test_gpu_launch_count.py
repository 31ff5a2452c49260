"""pfm_launch_count with two host threads (GPU test): the kernels of a fixed sequence
of calls are counted alike whether another thread works in the library meanwhile or
not, with V-cycles that replay a CUDA graph."""
import threading

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


def test_two_threads_count_every_launch_once(binding):
    ps, rs, streams = [], [], []
    for seed in (1, 2):
        st = inputs.config_random(9, 8, 8, seed=seed)
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            P = binding.problem_from_state(st)
            r = torch.from_numpy(st.U.astype("float32")).cuda()
        s.synchronize()
        P.set_stream(s)
        ps.append(P)
        rs.append(r)
        streams.append(s)
    opts = abi.default_opts(abi.PFM_F32)

    def work(k):
        torch.cuda.set_device(0)
        z = torch.empty_like(rs[k])
        for _ in range(30):
            ps[k].linearize(abi.PFM_F32)
            for _ in range(4):
                ps[k].vcycle(rs[k], z, opts)
        streams[k].synchronize()

    def count(run):
        c0 = binding.launch_count()
        run()
        return binding.launch_count() - c0

    for k in (0, 1):
        work(k)  # launch shapes tuned, graphs made
    alone = [count(lambda k=k: work(k)) for k in (0, 1)]
    assert alone == [count(lambda k=k: work(k)) for k in (0, 1)]

    def both():
        ts = [threading.Thread(target=work, args=(k,)) for k in (0, 1)]
        [t.start() for t in ts]
        [t.join() for t in ts]

    for _ in range(3):
        assert count(both) == sum(alone)
    [P.close() for P in ps]
