"""What times cover: a generated bank's kernel_ms includes the synthesis of its
templates, whenever it ran; the autotuner's probe of the 256-lag tile runs whole
tiles only, as long searches do; a histogram of many bins does not rule a call."""
import time

import numpy as np
import pytest

from paper_1802_01685_gb300 import bf, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__
    __graft_entry__.build()
    h = bf.bf_init()
    yield h
    bf.bf_destroy(h)


def test_kernel_time_covers_the_synthesis(ctx):
    """One chunk of 6144 templates against 200 lags: they are made in about 100 us
    (12.6 million samples) and correlated in a tenth of that."""
    fs, T = 2048.0, 1.0
    spec = synth.grid_spec([synth.POWERLAW], [synth.ASC], [T], 50.0, 900.0, 64, 96)
    stored = bf.bf_bank_create_grid(ctx, spec, fs, T, bf.BF_BANK_SPLIT_BF16)
    gen = bf.bf_bank_create_grid(ctx, spec, fs, T, bf.BF_BANK_GENERATED)
    x = np.random.default_rng(1).standard_normal(2048 + 200).astype(np.float32)

    def ms(bank):
        best = 1e9
        for _ in range(6):
            res = bf.bf_correlate(ctx, bank, [x], fs, bf.make_opts())
            best = min(best, bf.bf_result_info_get(res).kernel_ms)
            bf.bf_result_destroy(res)
        return best

    assert ms(gen) >= ms(stored) + 0.05
    bf.bf_bank_destroy(stored)
    bf.bf_bank_destroy(gen)


def test_autotuner_times_whole_tiles():
    """A fresh context's first BF16 search runs the probe: four launches of each
    shape and no second launch of halves."""
    ctx = bf.bf_init()
    try:
        fs, T = 2048.0, 1.0
        spec = synth.grid_spec([synth.LINEAR], [synth.ASC], [T], 50.0, 900.0, 24, 16)     # 384: three template tiles
        bank = bf.bf_bank_create_grid(ctx, spec, fs, T, bf.BF_BANK_SPLIT_BF16)
        x = np.random.default_rng(2).standard_normal(20000).astype(np.float32)

        def launches():
            n0 = bf.bf_kernel_launches()
            bf.bf_result_destroy(bf.bf_correlate(ctx, bank, [x], fs, bf.make_opts(precision="bf16")))
            return bf.bf_kernel_launches() - n0

        first, second = launches(), launches()
        assert first - second == 8, (first, second)
        bf.bf_bank_destroy(bank)
    finally:
        bf.bf_destroy(ctx)


def test_many_bins_for_few_templates(ctx):
    """The last kernel copies the histograms to host memory.  A million bins of 64
    templates are 4 MB, which the whole GPU writes in 20 us of an 80 us call; by
    the one block that 64 templates need they took 800."""
    fs = 2048.0
    spec = synth.grid_spec([synth.LINEAR], [synth.ASC], [1.0], 60.0, 480.0, 8, 8)
    bank = bf.bf_bank_create_grid(ctx, spec, fs, 1.0, bf.BF_BANK_SPLIT_BF16)
    x = np.random.default_rng(6).standard_normal(8192).astype(np.float32)

    def call(bins):
        best = 1e9
        for _ in range(12):
            t0 = time.perf_counter()
            res = bf.bf_correlate(ctx, bank, [x], fs, bf.make_opts(hist_bins=bins))
            best = min(best, time.perf_counter() - t0)
            out = bf.bf_result_copy_to_host(res, 0)
            bf.bf_result_destroy(res)
        want = np.bincount(np.minimum((out["max"] * np.float32(bins)).astype(np.int64), bins - 1), minlength=bins)
        np.testing.assert_array_equal(out["hist"], want)
        return best

    assert call(1_000_000) < 4.0 * call(1024)
    bf.bf_bank_destroy(bank)
