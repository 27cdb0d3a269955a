"""The host views show what launches run: the covers that contexts take, and the
split of a launch's work over the SMs, for one context and for several problems
of a batch (no GPU needed)."""
import random

import numpy as np
import pytest


@pytest.fixture(scope="module")
def corr():
    from paper_2406_19013_gb300 import build
    build.build()
    from paper_2406_19013_gb300 import corr as c
    return c


def _unit_channels(n_in):
    """Channels of a unit: two 64-row tiles of 64 / n16 channels up to 32
    inputs, two channels up to one row tile, otherwise one."""
    if n_in <= 32:
        return 2 * (64 // (-(-n_in // 16) * 16))
    return 2 if n_in <= 64 else 1


def _check(corr, shapes, n_blocks, grid):
    items, first = corr.plan_launch(shapes, n_blocks, grid)
    assert 1 <= len(first) - 1 <= grid
    assert first[0] == 0 and first[-1] == len(items) and np.all(np.diff(first) >= 1)
    for p, (n_in, n_chan, block_len) in enumerate(shapes):
        n_tpl = corr.plan(n_in)[0]
        npk, step = -(-block_len // 128) * n_blocks, _unit_channels(n_in)
        mine = items[items[:, 0] == p]
        assert np.all(mine[:, 2] % step == 0)
        assert mine[:, 3].min() >= 0 and mine[:, 4].min() >= 1
        assert (mine[:, 3] + mine[:, 4]).max() <= npk
        # an item folds once, and its fp32 partials are exact over this many samples
        assert mine[:, 4].max() <= corr.CORR_EXACT_SAMPLES // 128
        seen = np.zeros((n_tpl, -(-n_chan // step), npk), dtype=np.int32)
        for _, tpl, chan, pk0, n in mine:
            seen[tpl, chan // step, pk0:pk0 + n] += 1
        assert np.all(seen == 1)
    return items, first


@pytest.mark.parametrize("n_in", [1, 16, 17, 32, 33, 48, 64, 65, 100, 128])
def test_small_contexts_run_the_gram_form(corr, n_in):
    n16 = -(-n_in // 16) * 16
    n_units, issued, cover = corr.plan(n_in, with_cover=True)
    assert n_units == 1
    assert np.array_equal(cover, np.tril(np.ones((n_in, n_in), dtype=np.uint8)))
    # every row tile against its columns; up to 32 inputs a channel's share of
    # a tile of 64 rows x 64 columns
    want = (64 * 64 * n16 // 64 if n_in <= 32 else 64 * n16 if n_in <= 64
            else 64 * (64 + n16))
    assert issued == want
    # the view's items step by the channels of a unit
    items, _ = corr.plan_items(n_in, 9, 256, 1, 152)
    assert sorted(items[:, 2]) == list(range(0, 9, _unit_channels(n_in)))


@pytest.mark.parametrize("n_in,cover", [(192, 0), (256, 0), (257, 2), (1152, 2), (1153, 3), (2048, 3)])
def test_plan_shows_the_cover_that_contexts_run(corr, n_in, cover):
    assert corr.plan(n_in)[:2] == corr.plan_cover(n_in, cover)[:2]


def test_plan_follows_the_kernel_choice(corr, monkeypatch):
    monkeypatch.setenv("CORR_CMAC_KERNEL", "pair")
    assert corr.plan(300)[:2] == corr.plan_cover(300, corr.CORR_COVER_QUADS)[:2]
    monkeypatch.setenv("CORR_CMAC_KERNEL", "smem")
    assert corr.plan(2048)[:2] == corr.plan_cover(2048, corr.CORR_COVER_PAIRS)[:2]
    assert corr.plan(192)[:2] == corr.plan_cover(192, corr.CORR_COVER_WINDOW)[:2]


@pytest.mark.parametrize("n_in,n_chan,block_len,n_blocks,grid", [
    (16, 64, 2048, 1, 152), (1, 1, 1, 1, 152), (5, 9, 40, 8, 152), (32, 3, 300000, 1, 152),
    (48, 3, 33001, 1, 152), (64, 256, 4096, 1, 152), (75, 200, 3001, 1, 152), (100, 3, 4096, 2, 152),
    (128, 512, 8192, 4, 152), (150, 3, 192, 8, 152), (192, 100, 1536, 1, 152), (192, 1, 200001, 1, 152),
    (200, 7, 2064, 2, 152), (256, 2, 1040, 1, 152), (300, 40, 2112, 3, 152), (512, 2, 1024, 1, 152),
    (1200, 1, 192, 3, 76), (2048, 4, 4096, 4, 76), (64, 1, 16384, 1, 7), (64, 1, 8192, 1, 1)])
def test_context_launches_cover_every_unit_stage_once(corr, n_in, n_chan, block_len, n_blocks, grid):
    _check(corr, [(n_in, n_chan, block_len)], n_blocks, grid)


@pytest.mark.parametrize("seed", range(24))
def test_batch_launches_cover_every_unit_stage_once(corr, seed):
    rng = random.Random(seed)
    sizes = rng.choice([(1, 128), (129, 1152), (1153, 2048)])
    shapes = [(rng.randint(*sizes), rng.randint(1, 3 if sizes[1] > 1152 else 40),
               rng.choice([rng.randint(1, 64), rng.randint(1, 9000), rng.randint(30000, 200000)]))
              for _ in range(rng.randint(1, 6))]
    _check(corr, shapes, 1, 76 if sizes[1] > 1152 else rng.choice([1, 5, 152]))


def test_few_units_fill_the_sms(corr):
    # 8 units of 16 stages: run whole they would take 8 SMs
    _, first = _check(corr, [(16, 64, 2048)], 1, 152)
    assert len(first) - 1 == 128


@pytest.mark.parametrize("shapes,n_blocks,grid", [
    ([], 1, 152), ([(192, 4, 64)] * 129, 1, 152), ([(0, 4, 64)], 1, 152), ([(8193, 4, 64)], 1, 152),
    ([(192, 0, 64)], 1, 152), ([(192, 4, 0)], 1, 152), ([(192, 4, 16777216)], 1, 152),
    ([(192, 4, 64)], 0, 152), ([(192, 4, 64)], 9, 152), ([(192, 4, 64)], 1, 0),
    ([(64, 4, 64), (192, 4, 64)], 1, 152),     # Gram form and A/Q rows
    ([(192, 4, 64), (2048, 4, 64)], 1, 152)])  # one-CTA units and pairs
def test_plan_launch_rejects(corr, shapes, n_blocks, grid):
    with pytest.raises(corr.CorrError) as e:
        corr.plan_launch(shapes, n_blocks, grid)
    assert e.value.code == corr.CORR_EINVAL


def test_batch_launches_follow_the_kernel_choice(corr, monkeypatch):
    # 1280 inputs: 37 one-CTA templates against 15 of CTA pairs
    shape = [(1280, 2, 256)]
    pairs = corr.plan_cover(1280, corr.CORR_COVER_PAIRS)[0]
    quads = corr.plan_cover(1280, corr.CORR_COVER_QUADS)[0]
    assert corr.plan_launch(shape, 1, 76)[0][:, 1].max() + 1 == quads
    monkeypatch.setenv("CORR_CMAC_KERNEL", "smem")
    assert corr.plan_launch(shape, 1, 152)[0][:, 1].max() + 1 == pairs
    # =pair is for contexts alone
    monkeypatch.setenv("CORR_CMAC_KERNEL", "pair")
    assert (corr.plan_launch([(512, 2, 256)], 1, 76)[0][:, 1].max() + 1
            == corr.plan_cover(512, corr.CORR_COVER_QUADS)[0])
    assert (corr.plan_launch([(512, 2, 256)] * 2, 1, 76)[0][:, 1].max() + 1
            == corr.plan_cover(512, corr.CORR_COVER_PAIRS)[0])


def test_fold_window_keeps_every_partial_exact(corr):
    # the operands are v + 8 in [0, 15]: a sample adds up to 2 x 15 x 15 to an
    # accumulator, and fp32 holds every integer up to 2^24
    assert 2 * 15 * 15 * corr.CORR_EXACT_SAMPLES < 2**24


@pytest.mark.parametrize("cover", [0, 1, 2, 3])
@pytest.mark.parametrize("n_in,n_chan,block_len,n_blocks,grid", [
    (16, 3, 300000, 1, 152), (128, 2, 200001, 1, 152), (192, 4, 2000000, 1, 152),
    (256, 2, 131071, 1, 3), (300, 2, 65536, 2, 152), (512, 1, 32769, 3, 1), (1300, 1, 100000, 1, 76)])
def test_items_end_within_the_fold_window(corr, n_in, n_chan, block_len, n_blocks, grid, cover):
    window = corr.CORR_EXACT_SAMPLES // 128
    items, _ = corr.plan_items(n_in, n_chan, block_len, n_blocks, grid, cover)
    assert items[:, 4].max() <= window
    npk = -(-block_len // 128) * n_blocks
    per_unit = _unit_channels(n_in) if cover == 0 and n_in <= 256 else 1
    n_tpl = corr.plan_cover(n_in, cover)[0]
    assert len(items) >= n_tpl * -(-n_chan // per_unit) * -(-npk // window)
