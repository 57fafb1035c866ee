"""The FFT correlation kernel's division of the work: every CTA takes a
contiguous share of the (template, series, segment) items and its two groups
of threads take them in turn, handing the template's spectrum over from row to
row.  The cases put the hand-over where it can go wrong: one item in all, one
segment per row (every item another row), two and three (the group that
fetches alternates), a share that begins with a row's last segment, more rows
than CTAs, several series with one segment each.  Maxima, lags and sigma
against the FP64 oracle at the route's tolerance, plain and quadrature."""
import numpy as np
import pytest

import oracle
from paper_1802_01685_gb300 import bf, synth

from parity import TOL, check_maxima, check_sigma, oracle_params

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

FS, T = 1024.0, 0.25                     # M = 256: 16,129 lags a segment (pair route 7,937)


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__
    __graft_entry__.build()
    h = bf.bf_init()
    yield h
    bf.bf_destroy(h)


@pytest.mark.parametrize("quad", [False, True])
@pytest.mark.parametrize("I,J,lens", [
    (1, 1, [257]),                       # one item, two lags
    (1, 1, [20000]),                     # one row of two segments (pair route three)
    (1, 3, [300]),                       # three rows of one segment
    (31, 16, [400]),                     # 496 rows of one segment on 152 CTAs
    (31, 16, [20000]),                   # two (three) segments a row
    (19, 9, [300, 17000, 257]),          # four (five) segments in three series
    (7, 13, [40000, 5000, 5001, 33000]),
])
def test_shares_and_hand_over(ctx, quad, I, J, lens):
    spec = synth.grid_spec([synth.LINEAR], [synth.ASC], [T], 50.0, 500.0, I, J)
    storage = bf.BF_BANK_FP32 | (bf.BF_BANK_QUADRATURE if quad else 0)
    bank = bf.bf_bank_create_grid(ctx, spec, FS, T, storage)
    try:
        rng = np.random.default_rng(I * 1000 + J)
        xs = [rng.standard_normal(n).astype(np.float32) for n in lens]
        res = bf.bf_correlate(ctx, bank, xs, FS, bf.make_opts(precision="fft_fp32"))
        p = oracle_params(spec)
        for s, x in enumerate(xs):
            got = bf.bf_result_copy_to_host(res, s)
            ref = oracle.search(x, FS, p, 256, want_rho=True, quadrature=quad)
            check_maxima(got, ref, ref["rho"], TOL["fft_fp32"], f"series {s}")
            check_sigma(got, ref, TOL["fft_fp32"], f"series {s}")
        bf.bf_result_destroy(res)
    finally:
        bf.bf_bank_destroy(bank)
