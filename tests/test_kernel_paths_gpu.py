"""GPU parity at the edges of the kernels' variants: the biased operands' largest
values and fold windows, splits of few units, the allocation-free entry's units
and windows, pitched rows, and the dump's store widths.  Integer results: every
comparison is exact.
"""
import os

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

N_THREADS = max(1, min(os.cpu_count() or 1, 64))


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


@pytest.fixture(scope="module")
def corr(torch_cuda):
    from paper_2406_19013_gb300 import build
    build.build()
    from paper_2406_19013_gb300 import corr as c
    return c


def _vis(corr, torch, blocks, n_ant, n_pol, tcn=False):
    C, N, T = blocks[0].shape
    with corr.Correlator(n_ant, n_pol, C, T) as xc:
        for b in blocks:
            if tcn:
                b = np.ascontiguousarray(np.transpose(b, (2, 0, 1)))
                xc.push_block_tcn(torch.from_numpy(b).cuda())
            else:
                xc.push_block(torch.from_numpy(b).cuda())
        vis, _ = xc.dump()
        xc.check()
        return vis.cpu().numpy()


@pytest.mark.parametrize("tcn", [False, True])
@pytest.mark.parametrize("n_ant,C,T", [
    (8, 2, 33001),     # 7+7j runs past one fold window of 32768 samples
    (32, 3, 32768),    # exactly one window
    (24, 3, 33001),    # 48 inputs: two tiles of one channel each
    (64, 1, 32896),    # 128 inputs: two row tiles, two windows of unlike parity
    (80, 1, 40000),    # three row tiles
    (96, 2, 1024),
    (160, 1, 640),     # one-CTA units above 256 inputs
    (600, 1, 130),     # CTA pairs
])
def test_largest_operands(corr, torch_cuda, oracle_mod, n_ant, C, T, tcn):
    # u = 15 on both parts (7+7j) gives the largest biased products, u = 0
    # (-8-8j) the smallest; a random tail adds every value after a large sum
    N = 2 * n_ant
    rng = np.random.default_rng(T + N)
    x = rng.integers(0, 256, size=(C, N, T), dtype=np.uint8)
    x[:, : N // 2, : T - 64] = 0x77
    x[:, N // 2:, : T // 2] = 0x88
    got = _vis(corr, torch_cuda, [x], n_ant, 2, tcn)
    assert np.array_equal(got, oracle_mod.xcorr(x, n_threads=N_THREADS))


@pytest.mark.parametrize("n_ant,n_pol,C,T,nb", [
    (8, 2, 1, 8192, 1),      # one unit over 64 stages: equal pieces on many CTAs
    (2, 1, 9, 640, 3),       # tiles of four channels, five stages
    (50, 2, 3, 4096, 2),     # two-channel units, the last alone
    (96, 2, 100, 1536, 1),   # 100 units of 12 stages: finer cuts of the runs
    (100, 2, 7, 2064, 2),    # two templates
    (192, 2, 2, 1024, 1),    # several templates, channel by channel
    (577, 2, 1, 256, 2),     # CTA pairs (the smallest such count is 1153)
])
def test_launches_of_few_units(corr, torch_cuda, oracle_mod, synth_mod, n_ant, n_pol, C, T, nb):
    N = n_ant * n_pol
    blocks = [synth_mod.make_block(N, C, T, seed=900 + N, block=b) for b in range(nb)]
    got = _vis(corr, torch_cuda, blocks, n_ant, n_pol)
    want = None
    for b in blocks:
        want = oracle_mod.xcorr(b, vis=want, n_threads=N_THREADS)
    assert np.array_equal(got, want)


@pytest.mark.parametrize("N,C,T", [
    (5, 7, 16), (16, 9, 131056), (20, 5, 4096), (64, 11, 4096), (65, 3, 33008), (128, 3, 2048),
    (192, 3, 65536), (256, 2, 1040),
])
def test_static_entry_units_and_windows(corr, torch_cuda, oracle_mod, synth_mod, N, C, T):
    torch = torch_cuda
    x = synth_mod.make_block(N, C, T, seed=950 + N)
    x[:, :, : T // 2] = 0x77
    d = torch.from_numpy(x).cuda()
    vis = torch.full((C, N * (N + 1) // 2, 2), -1, dtype=torch.int64, device="cuda")
    corr.xcorr_static(d, N, 1, vis=vis)
    assert np.array_equal(vis.cpu().numpy(), oracle_mod.xcorr(x, n_threads=N_THREADS))


@pytest.mark.parametrize("T", [1, 2, 3, 5, 15, 17, 63, 130, 257])
@pytest.mark.parametrize("N", [1, 3, 66])
def test_pitched_rows(corr, torch_cuda, oracle_mod, N, T):
    rng = np.random.default_rng(T * 100 + N)
    x = rng.integers(0, 256, size=(3, N, T), dtype=np.uint8)
    got = _vis(corr, torch_cuda, [x], N, 1)
    assert np.array_equal(got, oracle_mod.xcorr(x))


@pytest.mark.parametrize("n_ant,C", [(1, 1), (2, 3), (33, 5), (96, 4)])
@pytest.mark.parametrize("offset", [0, 2])
def test_dump_into_stokes_of_either_alignment(corr, torch_cuda, oracle_mod, synth_mod, n_ant, C,
                                              offset):
    # offset 2: the Stokes output starts 16 bytes past a 32-byte boundary
    torch = torch_cuda
    N, T = 2 * n_ant, 64
    x = synth_mod.make_block(N, C, T, seed=970 + n_ant)
    n = C * (n_ant * (n_ant + 1) // 2) * 8
    store = torch.full((n + 4,), 7, dtype=torch.int64, device="cuda")
    with corr.Correlator(n_ant, 2, C, T) as xc:
        xc.push_block(torch.from_numpy(x).cuda())
        vis, st = xc.dump(stokes=store[offset:offset + n])
        xc.check()
    want = oracle_mod.xcorr(x)
    assert np.array_equal(vis.cpu().numpy(), want)
    assert np.array_equal(st.cpu().numpy().reshape(C, -1, 4, 2), oracle_mod.stokes(want, n_ant))
    assert (store[:offset] == 7).all() and (store[offset + n:] == 7).all()
