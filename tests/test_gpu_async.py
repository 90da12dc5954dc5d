"""The asynchronous one-block kernel (few columns per cluster): bit for bit the
two-block kernel in FP32 with Kp > 128, the oracle in FP64, and its bounded
waits."""
import numpy as np
import pytest

import oracle
from paper_2009_11742_gb300 import inputs
from test_gpu_cta import one_run, rom  # noqa: F401 (the fixture)

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# columns per cluster 1, 2, 3 and 4, ragged
# rows and last clusters, one step, steps around the forcing table's
# 32, few and many receivers (300 and more: tiles of 4 receivers, staged beyond 64 KB)
@pytest.mark.parametrize("Kv,Ks,M,R,N,r", [
    (129, 192, 1, 2, 33, 4), (192, 150, 40, 3, 64, 1), (256, 256, 9, 100, 31, 2), (200, 256, 31, 7, 70, 9),
    (512, 512, 7, 64, 40, 5), (512, 500, 14, 1, 1, 1), (512, 512, 27, 40, 65, 8), (512, 512, 28, 9, 40, 3),
    (384, 380, 25, 33, 36, 6),
    (256, 256, 1, 300, 12, 1), (250, 256, 30, 301, 9, 2), (512, 512, 3, 800, 6, 3)])
@pytest.mark.parametrize("form", ["ricker", "gauss1", "ftab", "xref"])
def test_async_bitwise_two_block(rom, Kv, Ks, M, R, N, r, form):
    p = inputs.make_problem(Kv, Ks, M, R, seed=Kv + M)
    h = rom.Rom.from_problem(p)
    assert h.plan(M)["variant"] == 1
    ftab = None
    if form == "gauss1":
        h.set_wavelet("gauss1")
    if form == "ftab":
        ftab = torch.as_tensor(np.random.default_rng(5).standard_normal((N, M)).astype(np.float32), device="cuda")
    if form == "xref":
        X = np.random.default_rng(6).standard_normal((Kv + Ks, M)) * 0.01
        h.set_reference(X[:Kv], None if M == 7 else X[Kv:])
    auto, two = (one_run(rom, h, p, k, N, r, ftab) for k in (0, 2))
    for a, b in zip(auto, two):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("Kv,Ks,M", [(1, 1, 3), (64, 60, 200), (130, 192, 50), (256, 250, 33)])
def test_async_f64(rom, Kv, Ks, M):
    """FP64, one to several columns per cluster, with and without a reference state."""
    N, r = 40, 3
    p = inputs.make_problem(Kv, Ks, M, 5, seed=M)
    h = rom.Rom.from_problem(p)
    V0, S0 = inputs.random_state(Kv, M, seed=1, scale=0.1), inputs.random_state(Ks, M, seed=2, scale=0.1)
    T = torch.as_tensor(p.T, dtype=torch.float64, device="cuda")
    for ref in (False, True):
        X = np.zeros((Kv + Ks, M))
        if ref:
            X = np.random.default_rng(6).standard_normal((Kv + Ks, M)) * 0.01
            h.set_reference(X[:Kv], X[Kv:])
        V, S = rom.Rom.new_state(Kv, M, "fp64", fill=V0), rom.Rom.new_state(Ks, M, "fp64", fill=S0)
        tr = torch.zeros((N // r, M, 5), dtype=torch.float64, device="cuda")
        h.run_rank2(V, S, T, N, r=r, traces=tr, prec="fp64")
        assert h.sync_status() == rom.ROM_OK
        Vo, So, tro = oracle.forward(p.Avs, p.Asv, p.g, p.C, p.dt, V0, S0, N, T=p.T, r=r,
                                     xref=(X[:Kv], X[Kv:]) if ref else None)
        # (the library's traces are records x M x R)
        for a, b in ((V, Vo), (S, So), (tr.transpose(1, 2), tro)):
            # sums of up to 256 products over 40 steps: about 40 x sqrt(256) roundings of 1.1e-16
            assert np.linalg.norm(a.cpu().numpy() - b) <= 1e-13 * np.linalg.norm(b)


# wider blocks: several column groups of 1, 2 and 4 columns, ragged last clusters,
# (M = 1100) more clusters than fit at once, and many receivers (tiles of 4, staged up to
# and beyond 64 KB, or, R = 1000, read from global memory)
@pytest.mark.parametrize("Kv,Ks,M,R,group", [
    (128, 128, 150, 7, 1), (128, 120, 200, 7, 2), (128, 128, 512, 7, 4), (256, 256, 269, 7, 2), (200, 256, 300, 7, 4),
    (256, 250, 1100, 7, 4), (60, 64, 500, 7, 4), (64, 64, 380, 7, 1), (128, 128, 150, 301, 1), (256, 256, 269, 300, 2),
    (60, 64, 500, 203, 4), (256, 250, 269, 1000, 2)])
def test_async_f64_several_groups(rom, Kv, Ks, M, R, group):
    N, r = 9, 2
    p = inputs.make_problem(Kv, Ks, M, R, seed=M)
    h = rom.Rom.from_problem(p)
    W = h.plan(M, "fp64")["cols_per_block"]
    # the planner's blocks are a multiple of 4, 2 or 1 columns for groups of as many
    assert W > group and {0: 4, 2: 2}.get(W % 4, 1) == group
    V0, S0 = inputs.random_state(Kv, M, seed=1, scale=0.1), inputs.random_state(Ks, M, seed=2, scale=0.1)
    V, S = rom.Rom.new_state(Kv, M, "fp64", fill=V0), rom.Rom.new_state(Ks, M, "fp64", fill=S0)
    tr = torch.zeros((N // r, M, R), dtype=torch.float64, device="cuda")
    h.run_rank2(V, S, torch.as_tensor(p.T, dtype=torch.float64, device="cuda"), N, r=r, traces=tr, prec="fp64")
    assert h.sync_status() == rom.ROM_OK
    Vo, So, tro = oracle.forward(p.Avs, p.Asv, p.g, p.C, p.dt, V0, S0, N, T=p.T, r=r)
    for a, b in ((V, Vo), (S, So), (tr.transpose(1, 2), tro)):
        a = a.cpu().numpy()
        # column by column; as above, with 9 steps
        num, den = np.linalg.norm(a - b, axis=-2), np.linalg.norm(b, axis=-2)
        assert np.all(num <= 1e-13 * den)


@pytest.mark.parametrize("Kv,M,prec", [(512, 20, "fp32"), (128, 16, "fp64")])
def test_async_wait_limit(rom, Kv, M, prec):
    """Waits that run out end the kernel with a status; the context stays usable."""
    p = inputs.make_problem(Kv, Kv, M, 0, seed=20)
    h = rom.Rom.from_problem(p)
    T = torch.as_tensor(p.T, dtype=torch.float64 if prec == "fp64" else torch.float32, device="cuda")

    def run():
        V, S = rom.Rom.new_state(Kv, M, prec), rom.Rom.new_state(Kv, M, prec)
        h.run_rank2(V, S, T, 100, prec=prec)
        return h.sync_status(), V.cpu().numpy()
    assert rom.rom_set_wait_limit(h.h, 2_000_000) == rom.ROM_OK  # about 1 ms
    assert rom.rom_debug_inject_stall(h.h, 1) == rom.ROM_OK
    assert run()[0] == rom.ROM_E_TIMEOUT
    assert rom.rom_debug_inject_stall(h.h, 0) == rom.ROM_OK
    assert rom.rom_set_wait_limit(h.h, 4_000_000_000) == rom.ROM_OK
    status, V = run()
    Z = np.zeros((Kv, M))
    Vo, _, _ = oracle.forward(p.Avs, p.Asv, p.g, None, p.dt, Z, Z, 100, T=p.T)
    assert status == rom.ROM_OK and np.linalg.norm(V - Vo) <= 1e-4 * np.linalg.norm(Vo)


@pytest.mark.parametrize("K", [64, 256, 400])
def test_fp64_and_rank1_refuse_a_two_block_pin(rom, K):
    """FP64 and rank-1 runs have no two-block kernel, whatever their size."""
    p = inputs.make_problem(K, K, 3, 0, seed=1)
    h = rom.Rom.from_problem(p)
    T = torch.as_tensor(p.T, dtype=torch.float64, device="cuda")
    for kernel in (rom.ROM_KERNEL_AUTO, rom.ROM_KERNEL_ONE_BLOCK, rom.ROM_KERNEL_TWO_BLOCK, rom.ROM_KERNEL_DATAFLOW):
        h.set_kernel(kernel)
        pinned = kernel in (rom.ROM_KERNEL_TWO_BLOCK, rom.ROM_KERNEL_DATAFLOW)
        V, S = rom.Rom.new_state(K, 3, "fp64"), rom.Rom.new_state(K, 3, "fp64")
        v, s = torch.zeros(K, device="cuda"), torch.zeros(K, device="cuda")
        for call in (lambda: h.run_rank2(V, S, T, 4, prec="fp64"), lambda: h.run_rank1(v, s, 30.0, 4)):
            if pinned:
                with pytest.raises(rom.RomError) as err:
                    call()
                assert err.value.status == rom.ROM_E_UNSUPPORTED
            else:
                call()
        assert h.sync_status() == rom.ROM_OK
