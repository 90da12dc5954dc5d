"""Threads that run the same kernels at different sizes, each on its own
stream: every call succeeds and gives what it gives alone."""
import threading

import numpy as np
import pytest

from paper_2009_11742_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rom():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2009_11742_gb300 import build
    build.build()
    from paper_2009_11742_gb300 import rom as R
    return R


def side_by_side(calls, times):
    """calls: functions of a stream that give the tensors of one result.  Each
    runs once alone, then `times` times on a thread and stream of its own beside
    the others."""
    main = torch.cuda.current_stream()
    alone = [[x.clone() for x in call(main)] for call in calls]
    torch.cuda.synchronize()
    errors, start = [], threading.Barrier(len(calls))

    def loop(call, ref):
        try:
            st = torch.cuda.Stream()
            with torch.cuda.stream(st):
                start.wait()
                for _ in range(times):
                    out = call(st)
                st.synchronize()
                assert all(torch.equal(x, y) for x, y in zip(out, ref))
        except Exception as e:
            errors.append(e)
    threads = [threading.Thread(target=loop, args=a) for a in zip(calls, alone)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors


def test_statistics_of_different_widths(rom):
    def call(M):
        x = torch.randn((2, M, 9), device="cuda")
        return lambda st: rom.trace_stats(x, stream=st)
    side_by_side([call(M) for M in (4096, 3000, 2200, 4000)], times=2000)


def test_full_order_models_of_different_sizes(rom):
    def call(Nr, Nt):
        f = rom.Fom(Nr, Nt, dt=0.01)
        X0 = [torch.randn(x.shape, device="cuda") for x in f.new_state(36)]

        def one(st):
            X = [x.clone() for x in X0]
            f.run(*X, 40)
            return X
        return one
    side_by_side([call(300, 64), call(4, 16), call(20, 30)], times=200)


@pytest.mark.parametrize("K", [128, 320])
def test_rank2_runs_of_different_widths(rom, K):
    def call(M, prec):
        p = inputs.make_problem(K, K, M, 0, seed=M)
        h = rom.Rom.from_problem(p)
        V0 = rom.Rom.new_state(K, M, prec, fill=inputs.random_state(K, M, seed=1, scale=0.1))
        T = torch.as_tensor(p.T.astype(np.float64 if prec == "fp64" else np.float32), device="cuda")

        def one(st):
            V, S = V0.clone(), V0.clone()
            h.run_rank2(V, S, T, 20, prec=prec)
            return V, S
        return one
    side_by_side([call(M, prec) for M, prec in ((30, "fp32"), (700, "fp32"), (300, "fp32"), (20, "fp64"),
                                                (200, "fp64"))], times=200)
