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


@pytest.mark.parametrize("tcn", [False, True])
@pytest.mark.parametrize("n_ant,C,T,nb", [
    (128, 2, 4160, 1),     # 256 inputs, 65 chunks a block, cut into equal pieces
    (128, 5, 64, 8),       # one chunk a block
    (150, 3, 192, 8),      # two operand stages, three chunks a block
    (150, 40, 2112, 3),    # the same, 33 chunks, every SM busy
    (96, 2, 320, 7),       # three operand stages, five chunks a block
    (96, 1, 40, 8),        # less than a chunk a block
    (40, 3, 192, 5),       # Gram form: a stage is a chunk
    (600, 1, 192, 3),      # CTA pairs
])
def test_odd_chunk_counts(corr, torch_cuda, oracle_mod, synth_mod, n_ant, C, T, nb, tcn):
    # blocks of an odd number of 64-sample chunks: the two unpack groups then
    # meet every block with changed turns
    N = 2 * n_ant
    blocks = [synth_mod.make_block(N, C, T, seed=930 + N, block=b) for b in range(nb)]
    torch = torch_cuda
    want = None
    for b in blocks:
        want = oracle_mod.xcorr(b, vis=want, n_threads=N_THREADS)
    with corr.Correlator(n_ant, 2, C, T) as xc:
        for _ in range(3):  # the same launches again: a race need not show at once
            if tcn:
                for b in blocks:
                    b = np.ascontiguousarray(np.transpose(b, (2, 0, 1)))
                    xc.push_block_tcn(torch.from_numpy(b).cuda())
            else:
                xc.push_blocks([torch.from_numpy(b).cuda() for b in blocks])
            vis, _ = xc.dump(want_stokes=False)
            xc.check()
            assert np.array_equal(vis.cpu().numpy(), want)


@pytest.mark.parametrize("seed", range(6))
def test_batches_of_few_uneven_units(corr, torch_cuda, oracle_mod, synth_mod, seed):
    # launch groups of several small instances, whose splits the search for a
    # shorter run changes
    torch = torch_cuda
    rng = np.random.default_rng(seed)
    shapes = [(n // 2, 2, int(rng.integers(1, 40)), 16 * int(rng.integers(1, 100)))
              for n in rng.choice([4, 32, 64, 100, 128, 192, 200, 256, 300], size=7)]
    blocks = [synth_mod.make_block(2 * a, c, t, seed=990 + seed, block=k)
              for k, (a, _, c, t) in enumerate(shapes)]
    with corr.Batch(shapes) as bt:
        for _ in range(2):
            bt.push([torch.from_numpy(x).cuda() for x in blocks])
        bt.check()
        for k, (a, _, _, _) in enumerate(shapes):
            vis, _ = bt.dump(k, want_stokes=False)
            want = 2 * oracle_mod.xcorr(blocks[k], n_threads=N_THREADS)
            assert np.array_equal(vis.cpu().numpy(), want), (k, shapes[k])


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


def _impulse_engine(corr, torch, n_spectra):
    # an impulse at the first sample of segment 2 is the centre tap of spectrum
    # 0: X[c] is the same real number for every channel, exactly (the DFT adds
    # zeros to it)
    adc = torch.zeros((1, (n_spectra + 3) * 2048), dtype=torch.int8, device="cuda")
    adc[0, 2 * 2048] = 100
    fe = corr.FEngine(1, n_spectra)
    fe.set_eq(np.ones((1, 1024), dtype=np.float32))
    x = fe.spectra(adc).cpu().numpy()[:, 0, 0]
    assert (x[:, 0] == x[0, 0]).all() and not x[:, 1].any()
    return adc, fe, np.float32(x[0, 0])


@pytest.mark.parametrize("n_spectra", [32, 5])
def test_fengine_codes_at_rounding_boundaries(corr, torch_cuda, n_spectra):
    # gains that bring X to every half-integer up to the clip, and to its
    # neighbours in fp32 on both sides; the code is the fp32 product rounded
    # half away from zero, clipped to [-7, 7]
    adc, fe, x0 = _impulse_engine(corr, torch_cuda, n_spectra)
    targets = [s * (k + h) for k in range(10) for h in (0.0, 0.5) for s in (1.0, -1.0)]
    g = [np.float32(t) / x0 for t in targets]
    for step in (1, 2, 3):
        for t in targets:
            lo = hi = np.float32(t) / x0
            for _ in range(step):
                lo, hi = np.nextafter(lo, np.float32(-np.inf)), np.nextafter(hi, np.float32(np.inf))
            g += [lo, hi]
    g += [np.float32(v) for v in (np.inf, -np.inf, np.nan, 1e30, -1e30, 1e-30, 0.0, -0.0)]
    eq = np.zeros((1, 1024), dtype=np.float32)
    eq[0, : len(g)] = g
    assert len(g) < 1024
    fe.set_eq(eq)
    codes = fe.run(adc).cpu().numpy()[:, 0, 0]
    with np.errstate(all="ignore"):
        re, im = eq[0] * x0, eq[0] * np.float32(0.0)
    for c in range(1024):
        want = 0
        for v, shift in ((re[c], 4), (im[c], 0)):
            if np.isnan(v):
                q = -7  # fmax(NaN, -7)
            else:
                q = int(np.sign(v) * np.floor(np.abs(np.float64(np.clip(v, -7, 7))) + 0.5))
            want |= (q & 15) << shift
        assert codes[c] == want, (c, eq[0, c], re[c])


@pytest.mark.parametrize("n_in,n_spectra", [(3, 64), (2, 32), (2, 96)])
def test_fengine_output_alignments(corr, torch_cuda, synth_mod, n_in, n_spectra):
    # rows in whole 32-byte stores, and the same output 16 bytes off
    torch = torch_cuda
    adc = torch.from_numpy(synth_mod.adc_streams(n_in, (n_spectra + 3) * 2048, seed=41)).cuda()
    n = 1024 * n_in * n_spectra
    store = torch.full((n + 64,), 0xAB, dtype=torch.uint8, device="cuda")
    with corr.FEngine(n_in, n_spectra, synth_mod.eq_for_noise(n_in, 20.0)) as fe:
        want = fe.run(adc)
        fe.run(adc, out=store[16:16 + n])
    assert torch.equal(store[16:16 + n], want.view(-1))
    assert (store[:16] == 0xAB).all() and (store[16 + n:] == 0xAB).all()


@pytest.mark.parametrize("n_in", [1, 3])
@pytest.mark.parametrize("n_spectra", [1, 2, 3, 4, 5, 8, 9, 15, 16, 17, 31, 33, 36, 47, 63])
def test_fengine_rows_of_any_length(corr, torch_cuda, synth_mod, n_in, n_spectra):
    # a spectrum's codes depend on its own samples alone: the first columns of
    # a run of whole tiles, with nothing written around them
    torch = torch_cuda
    whole = 64
    x = synth_mod.adc_streams(n_in, (whole + 3) * 2048, seed=43)
    eq = synth_mod.eq_for_noise(n_in, 20.0)
    with corr.FEngine(n_in, whole, eq) as fe:
        want = fe.run(torch.from_numpy(x).cuda())[:, :, :n_spectra]
    n = 1024 * n_in * n_spectra
    store = torch.full((n + 64,), 0xAB, dtype=torch.uint8, device="cuda")
    with corr.FEngine(n_in, n_spectra, eq) as fe:
        head = np.ascontiguousarray(x[:, : (n_spectra + 3) * 2048])
        fe.run(torch.from_numpy(head).cuda(), out=store[16:16 + n])
    assert torch.equal(store[16:16 + n].view(1024, n_in, n_spectra), want)
    assert (store[:16] == 0xAB).all() and (store[16 + n:] == 0xAB).all()


@pytest.mark.parametrize("N,C,T", [
    (1, 1, 16), (5, 9, 16), (16, 5, 128), (17, 3, 144), (32, 76, 128),   # tiles of several channels
    (33, 2, 16), (48, 7, 1024), (64, 1, 16), (64, 9, 256),               # one channel a tile
    (64, 76, 256), (64, 77, 256), (16, 608, 128), (16, 616, 128),        # both sides of the rule at 152 SMs
    (65, 1, 16), (128, 1, 128),                                          # two row tiles
])
def test_static_entry_on_few_units(corr, torch_cuda, oracle_mod, synth_mod, N, C, T):
    torch = torch_cuda
    x = synth_mod.make_block(N, C, T, seed=1010 + N)
    vis = torch.full((C + 1, N * (N + 1) // 2, 2), -1, dtype=torch.int64, device="cuda")
    corr.xcorr_static(torch.from_numpy(x).cuda(), N, 1, vis=vis)
    got = vis.cpu().numpy()
    assert np.array_equal(got[:C], oracle_mod.xcorr(x, n_threads=N_THREADS))
    assert (got[C] == -1).all()
