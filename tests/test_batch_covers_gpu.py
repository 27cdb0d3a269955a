"""The covers that a batch's instances run, as corr_batch_info reports them."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SHAPES = [(600, 2, 2, 192), (150, 2, 3, 192), (16, 2, 5, 256)]  # 1200, 300 and 32 inputs


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


def _covers(corr, torch, oracle_mod, synth_mod, autotune=False):
    blocks = [synth_mod.make_block(a * p, c, t, seed=70, block=k)
              for k, (a, p, c, t) in enumerate(SHAPES)]
    with corr.Batch(SHAPES, autotune=autotune) as bt:
        bt.push([torch.from_numpy(x).cuda() for x in blocks])
        bt.check()
        for k, x in enumerate(blocks):
            vis, _ = bt.dump(k, want_stokes=False)
            assert np.array_equal(vis.cpu().numpy(), oracle_mod.xcorr(x)), SHAPES[k]
        return [bt.info(k)[0] for k in range(len(SHAPES))]


@pytest.mark.parametrize("autotune", [False, True])
def test_info_reports_the_cover_that_runs(corr, torch_cuda, oracle_mod, synth_mod, autotune):
    got = _covers(corr, torch_cuda, oracle_mod, synth_mod, autotune)
    assert got[:2] == [corr.CORR_COVER_QUADS, corr.CORR_COVER_PAIRS]
    if autotune:
        assert [corr.tuned_cover(a * p, t) for a, p, _, t in SHAPES] == got
    else:
        assert got[2] == corr.CORR_COVER_WINDOW


@pytest.mark.parametrize("autotune", [False, True])
def test_one_cta_units_can_be_asked_for(corr, torch_cuda, oracle_mod, synth_mod, monkeypatch,
                                        autotune):
    # CTA pairs above 1152 inputs are a default, for batches as for contexts
    monkeypatch.setenv("CORR_CMAC_KERNEL", "smem")
    got = _covers(corr, torch_cuda, oracle_mod, synth_mod, autotune)
    assert got[:2] == [corr.CORR_COVER_PAIRS, corr.CORR_COVER_PAIRS]
