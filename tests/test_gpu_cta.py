"""The one-CTA rank-2 kernel (FP32, Kp <= 128, the planner's choice for small
models) against the two-block split kernel, whose sums, reduction, epilogue
and traces it repeats: every result is equal bit for bit (the split kernel is
itself held to the FP64 oracle)."""
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


def one_run(rom, h, p, kernel, N, r, ftab=None, n0=3):
    h.set_kernel(kernel)
    Kv, Ks, M = p.Kv, p.Ks, p.M
    V = rom.Rom.new_state(Kv, M, "fp32", fill=inputs.random_state(Kv, M, seed=1, scale=0.1))
    S = rom.Rom.new_state(Ks, M, "fp32", fill=inputs.random_state(Ks, M, seed=2, scale=0.1))
    cV = rom.Rom.new_state(Kv, M, "fp32", fill=inputs.random_state(Kv, M, seed=3, scale=1e-9))
    cS = rom.Rom.new_state(Ks, M, "fp32", fill=inputs.random_state(Ks, M, seed=4, scale=1e-9))
    T = torch.as_tensor(p.T, device="cuda") if ftab is None else None
    tr = torch.zeros((N // r, M, p.R), device="cuda") if r else None
    h.run_rank2(V, S, T, N, n0=n0, r=r, traces=tr, prec="fp32", compV=cV, compS=cS, ftab=ftab)
    torch.cuda.synchronize()
    assert h.sync_status() == 0
    return [x.cpu().numpy() for x in (V, S, cV, cS) + ((tr,) if r else ())]


# (Kv, Ks, M, R, N, r): both Kp, every column group, one block and several,
# more blocks than SMs, steps on both sides of the forcing table's length,
# receiver rows staged and (R = 200 at Kp = 128) read from global memory, and many
# receivers of one column (8 x 1 tiles: R = 77 and more)
@pytest.mark.parametrize("Kv,Ks,M,R,N,r", [
    (1, 1, 1, 0, 1, 0), (64, 64, 1, 1, 33, 1), (63, 2, 2, 5, 31, 2), (17, 40, 3, 64, 32, 3), (64, 50, 305, 3, 40, 7),
    (30, 64, 1300, 2, 20, 20), (65, 65, 1, 9, 65, 5), (128, 128, 2, 3, 64, 64), (100, 90, 5, 3, 50, 5),
    (90, 128, 153, 4, 30, 9), (128, 127, 460, 200, 12, 4), (66, 128, 1100, 1, 9, 3),
    (64, 64, 1, 200, 12, 4), (128, 120, 1, 77, 12, 1), (100, 128, 150, 130, 6, 2)])
@pytest.mark.parametrize("form", ["ricker", "gauss1", "ftab", "xref"])
def test_cta_bitwise_split(rom, Kv, Ks, M, R, N, r, form):
    p = inputs.make_problem(Kv, Ks, M, R, seed=Kv + M)
    h = rom.Rom.from_problem(p)
    assert h.plan(M)["variant"] == 5
    ftab = None
    if form == "gauss1":
        h.set_wavelet("gauss1")
    if form == "ftab":
        ftab = torch.as_tensor(np.random.default_rng(5).standard_normal((N, M)).astype(np.float32), device="cuda")
    if form == "xref":
        X = np.random.default_rng(6).standard_normal((Kv + Ks, M)) * 0.01
        h.set_reference(X[:Kv], None if M == 2 else X[Kv:])
    auto, split = (one_run(rom, h, p, k, N, r, ftab) for k in (0, 2))
    for a, b in zip(auto, split):
        assert np.array_equal(a, b)


def test_cta_nonfinite_status(rom):
    """A state that holds an infinity is reported as by the cluster kernels."""
    p = inputs.make_problem(40, 40, 3, 0, seed=9)
    h = rom.Rom.from_problem(p)
    V, S = rom.Rom.new_state(40, 3, "fp32"), rom.Rom.new_state(40, 3, "fp32")
    V[3, 1] = float("inf")
    h.run_rank2(V, S, torch.as_tensor(p.T, device="cuda"), 5)
    assert h.sync_status() == rom.ROM_E_NONFINITE
