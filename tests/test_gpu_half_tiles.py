"""Few 256-lag tiles run in halves of 128 lags on two SMs.  A series searched
alone (halves) and in a batch that fills the GPU (whole tiles) must give the
same maxima, lags and tails bit for bit, at lag counts around the half's and
the tile's edge, for every tensor-core precision, plain and quadrature; and the
search alone matches the oracle."""
import numpy as np
import pytest

import oracle
from paper_1802_01685_gb300 import bf, synth

from parity import TOL, check_maxima, check_sigma, oracle_params

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

FS, T, M = 2048.0, 1.0, 2048


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__
    __graft_entry__.build()
    h = bf.bf_init()
    yield h
    bf.bf_destroy(h)


@pytest.mark.parametrize("quad", [False, True])
@pytest.mark.parametrize("prec", ["split_bf16", "split_fp16", "bf16"])
def test_halves_equal_whole_tiles(ctx, prec, quad):
    spec = synth.grid_spec([synth.LINEAR], [synth.ASC, synth.DESC], [T, 0.5], 50.0, 900.0, 5, 8)      # 160 templates
    storage = (bf.BF_BANK_SPLIT_FP16 if prec == "split_fp16" else bf.BF_BANK_SPLIT_BF16)
    bank = bf.bf_bank_create_grid(ctx, spec, FS, T, storage | (bf.BF_BANK_QUADRATURE if quad else 0))
    rng = np.random.default_rng(3)
    lags = [1, 127, 128, 129, 255, 256, 257, 385, 700]
    xs = [rng.standard_normal(M - 1 + n).astype(np.float32) for n in lags]
    # the batch's first tiles are the short series', in whole rounds of one tile per
    # SM; alone each has at most 9, in halves
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    fill = rng.standard_normal(M - 1 + 2 * n_sm * 256).astype(np.float32)
    tt = -(-(2 if quad else 1) * 160 // 128)                  # template tiles
    tiles = [-(-n // 256) * tt for n in lags]
    assert 2 * max(tiles) <= n_sm and (sum(tiles) + 2 * n_sm * tt) // n_sm * n_sm >= sum(tiles)
    opts = bf.make_opts(precision=prec, want_tails=True, kappa=3.0, tile_lags=256)
    try:
        batch = bf.bf_correlate(ctx, bank, xs + [fill], FS, opts)
        assert bf.bf_result_info_get(batch).tile_lags == 256
        tails = bf.bf_result_copy_tails(batch)
        for s, x in enumerate(xs):
            alone = bf.bf_correlate(ctx, bank, [x], FS, opts)
            assert bf.bf_result_info_get(alone).tile_lags == 256
            a, b = bf.bf_result_copy_to_host(alone, 0), bf.bf_result_copy_to_host(batch, s)
            np.testing.assert_array_equal(a["max"], b["max"], err_msg=f"{lags[s]} lags")
            np.testing.assert_array_equal(a["argmax"], b["argmax"], err_msg=f"{lags[s]} lags")
            np.testing.assert_allclose(a["sigma"], b["sigma"], rtol=1e-6)
            ta = np.sort(bf.bf_result_copy_tails(alone), order=["k", "tau"])
            tb = np.sort(tails[tails["series"] == s], order=["k", "tau"])
            for f in ("k", "tau", "rho"):
                np.testing.assert_array_equal(ta[f], tb[f])
            if s in (3, 8):
                ref = oracle.search(x, FS, oracle_params(spec), M, want_rho=True, quadrature=quad)
                check_maxima(a, ref, ref["rho"], TOL[prec], f"{lags[s]} lags")
                check_sigma(a, ref, TOL[prec], f"{lags[s]} lags")
            bf.bf_result_destroy(alone)
        bf.bf_result_destroy(batch)
    finally:
        bf.bf_bank_destroy(bank)
