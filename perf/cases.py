"""The work that a user of this X-engine has it do, as cases that can be timed.

A case is one pass through the package's public entry points on device-resident data: an integration (blocks
pushed, then the dump with visibilities and, for dual-polarisation arrays, Stokes products), a batch of correlators,
the allocation-free call, or a run of the F-engine.  Sizes are those of the repository's own workloads (the paper's
192-input array, its batched, served and large-N configurations, their channel bands) and of its ragged tests.
"""
import math
import random

import torch

from paper_2406_19013_gb300 import corr as xg

P = 2048         # F-engine: points of the filter bank and FFT
TAPS = 4
CHANNELS = P // 2
TWO_PI = 2.0 * math.pi

# Input counts a batch cycles through (the batched workload's arrays).
BATCH_INPUTS = (32, 64, 128, 192, 256, 512)


def listed():
    return [
        # The smallest call: 8 dual-polarisation antennas, 64 channels, one block, dumped at once.  Latency and launches.
        dict(name="tiny_16in", kind="push", n_ant=8, n_pol=2, n_chan=64, block_len=2048, n_blocks=1),
        # A single-polarisation array of odd size with a block length that is no multiple of 16 bytes (rows are re-pitched).
        dict(name="ragged_75in_monopol", kind="push", n_ant=75, n_pol=1, n_chan=200, block_len=3001, n_blocks=3),
        # The allocation-free entry point on a mid-size array (code inside a framework that owns the device memory).
        dict(name="static_64in", kind="static", n_ant=32, n_pol=2, n_chan=256, block_len=4096),
        # A mid-size served array: 64 dual-polarisation antennas, four blocks to an integration.
        dict(name="array_128in", kind="push", n_ant=64, n_pol=2, n_chan=512, block_len=8192, n_blocks=4),
        # The paper's array at full band: 96 dual-polarisation antennas, 1024 channels, eight 8192-sample blocks, then the dump.
        dict(name="paper_192in", kind="push", n_ant=96, n_pol=2, n_chan=1024, block_len=8192, n_blocks=8),
        # The same array with a fast dump (about 8 ms of sky): the fold, visibilities and Stokes weigh as much as the products.
        dict(name="paper_fast_dump", kind="push", n_ant=96, n_pol=2, n_chan=1024, block_len=1024, n_blocks=1),
        # The same array with the block in the F-engine's order, [time][channel][input], turned while it is integrated.
        dict(name="paper_tcn", kind="tcn", n_ant=96, n_pol=2, n_chan=1024, block_len=4096, n_blocks=2),
        # The largest served array: 256 dual-polarisation antennas.
        dict(name="array_512in", kind="push", n_ant=256, n_pol=2, n_chan=128, block_len=8192, n_blocks=2),
        # Large N: 1024 dual-polarisation antennas, one of eight channel bands of the 256-channel configuration.
        dict(name="large_2048in", kind="push", n_ant=1024, n_pol=2, n_chan=32, block_len=4096, n_blocks=4),
        # Many correlators of uneven size in shared launches: the batched workload's draws on fewer instances.
        dict(name="batch_12", kind="batch", n_inst=12, shapes_seed=3, max_chan=256, max_len=8192),
        # The F-engine on the paper's array: 192 streams, 8192 spectra, codes in the X-engine's order.
        dict(name="fengine_192in", kind="fengine", n_in=192, n_spectra=8192),
        # A small F-engine run of odd size: few streams, a spectrum count that fills no whole tile.
        dict(name="fengine_17in", kind="fengine", n_in=17, n_spectra=1003),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))))


def _cost(n_in, n_chan, samples):
    """Complex products of an integration, rows padded to whole 64-input tiles (what small arrays cost in earnest)."""
    rows = 64 * ((n_in + 63) // 64)
    return rows * (rows + 64) // 2 * n_chan * samples


def draw(rng):
    """One more case: any array from 2 to 2048 inputs, any band and block length that costs no more than the paper's."""
    most = _cost(192, 1024, 8 * 8192)
    while True:
        kind = rng.choice(["push", "push", "push", "tcn", "static", "batch", "fengine"])
        if kind == "fengine":
            return dict(kind=kind, n_in=_log_int(rng, 1, 192), n_spectra=_log_int(rng, 33, 8192))
        if kind == "batch":
            return dict(kind=kind, n_inst=rng.randint(3, 12), shapes_seed=rng.randint(10, 10**6), max_chan=rng.randint(64, 256),
                        max_len=rng.randint(1024, 8192))
        n_pol = rng.choice([1, 2, 2])
        n_ant = _log_int(rng, 2, (256 if kind == "static" else 2048) // n_pol)
        if kind == "tcn" and rng.random() < 0.7:  # F-engine boards bring inputs in multiples of 16
            n_ant = max(16 // n_pol, n_ant * n_pol // 16 * 16 // n_pol)
        n_in = n_ant * n_pol
        n_chan, block_len = _log_int(rng, 8, 1024), _log_int(rng, 256, 16384)
        if kind == "static" or rng.random() < 0.6:  # most recorders pad their rows
            block_len = max(256, block_len // 16 * 16)
        n_blocks = 1 if kind == "static" else _log_int(rng, 1, 8)
        vis_bytes = n_chan * n_in * (n_in + 1) * 8
        # blocks that are turned or re-pitched first cost more for each product
        share = 4 if kind == "tcn" or block_len % 16 else 1
        if share * _cost(n_in, n_chan, block_len * n_blocks) <= most and vis_bytes <= 2.5e9 and n_in * n_chan * block_len <= 1.7e9:
            case = dict(kind=kind, n_ant=n_ant, n_pol=n_pol, n_chan=n_chan, block_len=block_len)
            return case if kind == "static" else dict(case, n_blocks=n_blocks)


def _batch_shapes(case):
    """(n_ant, n_pol, n_chan, block_len) of a batch's instances: uneven channel counts, block lengths on a 16-sample grid."""
    rng = random.Random(case["shapes_seed"])
    return [(BATCH_INPUTS[k % len(BATCH_INPUTS)] // 2, 2, rng.randint(16, case["max_chan"]), 16 * rng.randint(16, case["max_len"] // 16))
            for k in range(case["n_inst"])]


def _voltages(n_chan, n_in, n_time, gen, tcn=False):
    """uint8 voltages: Gaussian noise (sigma 2.5 per component) and a tone of amplitude 2 with a random phase per input,
    rounded and clipped to [-7, 7], the real part in the high nibble; [channel][input][time], or [time][channel][input]."""
    shape = (n_time, n_chan, n_in) if tcn else (n_chan, n_in, n_time)
    out = torch.empty(shape, dtype=torch.uint8, device="cuda")
    phase = torch.rand(n_in, generator=gen, device="cuda") * TWO_PI
    tone_re, tone_im = 2.0 * torch.cos(phase), 2.0 * torch.sin(phase)
    if not tcn:
        tone_re, tone_im = tone_re[:, None], tone_im[:, None]
    step = max(1, int(2**26 // (out.numel() // shape[0])))
    for lo in range(0, shape[0], step):
        part = out[lo:lo + step]
        re = torch.randn(part.shape, generator=gen, device="cuda").mul_(2.5).add_(tone_re).round_().clamp_(-7, 7).to(torch.int8)
        im = torch.randn(part.shape, generator=gen, device="cuda").mul_(2.5).add_(tone_im).round_().clamp_(-7, 7).to(torch.int8)
        part.copy_(re.bitwise_left_shift_(4).bitwise_or_(im.bitwise_and_(15)).view(torch.uint8))
    return out


def _generator(seed, salt=0):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed * 1000003 + salt)
    return gen


def _ring(case, seed):
    """The distinct blocks that a device-resident ring holds: at most two, pushed in turn."""
    n_in = case["n_ant"] * case["n_pol"]
    return [_voltages(case["n_chan"], n_in, case["block_len"], _generator(seed, k), tcn=case["kind"] == "tcn")
            for k in range(min(2, case.get("n_blocks", 1)))]


def _adc(n_in, n_samples, gen):
    """int8 samples: Gaussian noise of sigma 20 counts and a sinusoid of amplitude 8 at a channel centre."""
    out = torch.empty((n_in, n_samples), dtype=torch.int8, device="cuda")
    phase = torch.rand(n_in, generator=gen, device="cuda") * TWO_PI
    t = torch.arange(n_samples, device="cuda") % P
    for k in range(n_in):
        x = torch.randn(n_samples, generator=gen, device="cuda").mul_(20.0)
        x += 8.0 * torch.cos(t * (TWO_PI * 300 / P) + phase[k])
        out[k] = x.round_().clamp_(-128, 127).to(torch.int8)
    return out


def _prototype():
    m = torch.arange(TAPS * P, dtype=torch.float64)
    return (0.54 - 0.46 * torch.cos(TWO_PI * m / (TAPS * P - 1))) * torch.sinc((m - TAPS * P / 2) / P)


def _eq(n_in):
    """Gains that bring noise of sigma 20 to 2.5 per component, flattening a pass band with a gentle slope: float32[n_in][1024]."""
    g = 2.5 / (20.0 * math.sqrt(float((_prototype() ** 2).sum()) / 2.0))
    slope = 1.0 + 0.1 * torch.linspace(-1.0, 1.0, CHANNELS, dtype=torch.float64)
    return (g * slope).repeat(n_in, 1).to(torch.float32)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "fengine":
        n_in, n_spectra = case["n_in"], case["n_spectra"]
        return dict(case=case, engine=xg.FEngine(n_in, n_spectra, _eq(n_in).numpy()),
                    adc=_adc(n_in, (n_spectra + TAPS - 1) * P, _generator(seed)),
                    out=torch.empty((CHANNELS, n_in, n_spectra), dtype=torch.uint8, device="cuda"))
    if kind == "batch":
        shapes = _batch_shapes(case)
        outs = [(torch.empty((c, a * p * (a * p + 1) // 2, 2), dtype=torch.int64, device="cuda"),
                 torch.empty((c, a * (a + 1) // 2, 4, 2), dtype=torch.int64, device="cuda")) for a, p, c, _ in shapes]
        return dict(case=case, batch=xg.Batch(shapes), outs=outs,
                    blocks=[_voltages(c, a * p, t, _generator(seed, k)) for k, (a, p, c, t) in enumerate(shapes)])
    n_ant, n_pol, n_chan = case["n_ant"], case["n_pol"], case["n_chan"]
    n_in = n_ant * n_pol
    state = dict(case=case, blocks=_ring(case, seed),
                 vis=torch.empty((n_chan, n_in * (n_in + 1) // 2, 2), dtype=torch.int64, device="cuda"))
    if kind != "static":
        state["xc"] = xg.Correlator(n_ant, n_pol, n_chan, case["block_len"])
        state["stokes"] = torch.empty((n_chan, n_ant * (n_ant + 1) // 2, 4, 2), dtype=torch.int64, device="cuda") if n_pol == 2 else None
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "fengine":
        return state["engine"].run(state["adc"], out=state["out"])
    if kind == "batch":
        state["batch"].push(state["blocks"])
        return [list(state["batch"].dump(k, vis=v, stokes=s)) for k, (v, s) in enumerate(state["outs"])]
    blocks = state["blocks"]
    if kind == "static":
        return xg.xcorr_static(blocks[0], case["n_ant"], case["n_pol"], vis=state["vis"])
    xc = state["xc"]
    if kind == "tcn":
        for k in range(case["n_blocks"]):
            xc.push_block_tcn(blocks[k % len(blocks)])
    elif case["n_blocks"] == 1:
        xc.push_block(blocks[0])
    else:
        xc.push_blocks([blocks[k % len(blocks)] for k in range(case["n_blocks"])])
    vis, stokes = xc.dump(vis=state["vis"], stokes=state["stokes"])
    return [vis] if stokes is None else [vis, stokes]


def _integration_work(n_ant, n_pol, n_chan, samples, stokes):
    n_in = n_ant * n_pol
    out = n_chan * n_in * (n_in + 1) * 8 + (n_chan * n_ant * (n_ant + 1) * 32 if stokes else 0)
    return n_in * n_chan * samples + out, 8 * (n_in * (n_in + 1) // 2) * n_chan * samples


def work(case):
    kind = case["kind"]
    if kind == "fengine":
        n_in, n_spectra = case["n_in"], case["n_spectra"]
        # filter 2 TAPS P, 1024-point complex FFT 5 N log2 N, split and gain 8 per channel
        flops = (2 * TAPS * P + 5 * CHANNELS * 10 + 8 * CHANNELS) * n_in * n_spectra
        return {"bytes": n_in * (n_spectra + TAPS - 1) * P + CHANNELS * n_in * n_spectra + 4 * n_in * CHANNELS, "flops": flops}
    if kind == "batch":
        both = [_integration_work(a, p, c, t, True) for a, p, c, t in _batch_shapes(case)]
        return {"bytes": sum(b for b, _ in both), "flops": sum(f for _, f in both)}
    b, f = _integration_work(case["n_ant"], case["n_pol"], case["n_chan"], case["block_len"] * case.get("n_blocks", 1),
                             kind != "static" and case["n_pol"] == 2)
    return {"bytes": b, "flops": f}


def _visibilities(block, weight, tcn, vis):
    """Adds weight x the block's lower-triangle visibilities, from float64 products (every sum is a whole number below 2^53)."""
    n_chan, n_in = vis.shape[0], block.shape[2] if tcn else block.shape[1]
    i, j = torch.tril_indices(n_in, n_in, device="cuda")
    n_time = block.shape[0] if tcn else block.shape[2]
    step = max(1, int(2**27 // (n_in * n_time + n_in * n_in)))
    for lo in range(0, n_chan, step):
        x = block[:, lo:lo + step].permute(1, 2, 0) if tcn else block[lo:lo + step]
        x = x.contiguous().view(torch.int8)
        re = (x >> 4).to(torch.float64)
        im = ((x << 4) >> 4).to(torch.float64)
        v_re = torch.baddbmm(re @ re.mT, im, im.mT)
        v_im = torch.baddbmm(im @ re.mT, re, im.mT, alpha=-1)
        vis[lo:lo + step, :, 0] += weight * v_re[:, i, j].to(torch.int64)
        vis[lo:lo + step, :, 1] += weight * v_im[:, i, j].to(torch.int64)


def _stokes(vis, n_ant):
    p, q = torch.tril_indices(n_ant, n_ant, device="cuda")

    def pair(a, b):  # the visibility of inputs a >= b
        return vis[:, a * (a + 1) // 2 + b]

    xx, yy, yx = pair(2 * p, 2 * q), pair(2 * p + 1, 2 * q + 1), pair(2 * p + 1, 2 * q)
    xy = pair(torch.maximum(2 * p, 2 * q + 1), torch.minimum(2 * p, 2 * q + 1)).clone()
    xy[:, p == q, 1] *= -1  # above the diagonal: the conjugate
    out = torch.empty((vis.shape[0], p.numel(), 4, 2), dtype=torch.int64, device="cuda")
    out[:, :, 0], out[:, :, 1], out[:, :, 2] = xx + yy, xx - yy, xy + yx
    d = xy - yx
    out[:, :, 3, 0], out[:, :, 3, 1] = d[..., 1], -d[..., 0]
    return out


def _exact_codes(case, seed):
    n_in, n_spectra = case["n_in"], case["n_spectra"]
    adc = _adc(n_in, (n_spectra + TAPS - 1) * P, _generator(seed))
    h = _prototype().cuda().view(TAPS, P)
    eq = _eq(n_in).cuda().to(torch.float64)
    out = torch.empty((CHANNELS, n_in, n_spectra), dtype=torch.uint8, device="cuda")

    def code(v):
        return (torch.sign(v) * torch.floor(v.abs() + 0.5)).clamp(-7, 7).to(torch.int32)

    for k in range(n_in):
        x = adc[k].to(torch.float64).view(n_spectra + TAPS - 1, P)
        v = sum(h[j] * x[j:j + n_spectra] for j in range(TAPS))
        spec = torch.fft.rfft(v, dim=1)[:, :CHANNELS] * eq[k]
        out[:, k] = ((code(spec.real) << 4 & 0xF0) | (code(spec.imag) & 15)).to(torch.uint8).T
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "fengine":
        return _exact_codes(case, seed)
    if kind == "batch":
        outs = []
        for k, (a, p, c, t) in enumerate(_batch_shapes(case)):
            vis = torch.zeros((c, a * p * (a * p + 1) // 2, 2), dtype=torch.int64, device="cuda")
            _visibilities(_voltages(c, a * p, t, _generator(seed, k)), 1, False, vis)
            outs.append([vis, _stokes(vis, a)])
        return outs
    n_in, n_chan, n_blocks = case["n_ant"] * case["n_pol"], case["n_chan"], case.get("n_blocks", 1)
    ring = min(2, n_blocks)
    if 8.0 * n_in * n_in * n_chan * case["block_len"] * ring > 1.2e13:  # over about 20 seconds in float64
        return None
    vis = torch.zeros((n_chan, n_in * (n_in + 1) // 2, 2), dtype=torch.int64, device="cuda")
    for k, block in enumerate(_ring(case, seed)):
        _visibilities(block, len(range(k, n_blocks, ring)), kind == "tcn", vis)
    if kind == "static":
        return vis
    return [vis, _stokes(vis, case["n_ant"])] if case["n_pol"] == 2 else [vis]
