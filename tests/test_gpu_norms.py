"""Window norms where the FP64 prefix of x^2 is hard pressed: quiet data before
loud data (a prefix that took its own part off a total again would carry the
later samples' rounding), and series whose block sums take several rounds of
the scan.  Dense rho, maxima and sigma against the FP64 oracle."""
import numpy as np
import pytest

import oracle
from paper_1802_01685_gb300 import bf, synth

from parity import STORE_ALL, TOL, check_maxima, check_sigma, oracle_params, run

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__
    __graft_entry__.build()
    h = bf.bf_init()
    yield h
    bf.bf_destroy(h)


@pytest.mark.parametrize("loud", ["1e7", "1e8", "spike"])
def test_quiet_before_loud(ctx, loud):
    """A bank template in noise up to sample 6000, then data `loud` times
    louder, or one late sample of 1e9.  Every window before it has the norm of
    its own samples: none of the later energy may reach the prefix there."""
    fs, M = 2048.0, 2048
    spec = synth.grid_spec([synth.LINEAR, synth.POWERLAW], [synth.ASC, synth.DESC], [1.0, 0.4], 40.0, 900.0, 4, 4)
    bank = bf.bf_bank_create_grid(ctx, spec, fs, 1.0, STORE_ALL)
    p = oracle_params(spec)
    rng = np.random.default_rng(83)
    x = rng.standard_normal(8192)
    x[3200:3200 + M] += 200.0 * oracle.template(int(p["track"][5]), int(p["sense"][5]), p["f_lo"][5], p["f_hi"][5],
                                                p["D"][5], fs, M, 0)
    if loud == "spike":
        x[6500] = 1e9
    else:
        x[6000:] *= float(loud)
    x = x.astype(np.float32)
    ref = oracle.search(x, fs, p, M, want_rho=True)
    K, L = ref["rho"].shape
    # Split-FP16 scales the largest sample (here about 4 times `loud`) below 2^14
    # and has a spacing of 2^-24 there: noise of 1 is held to 4 loud 2^-38 / sqrt(3)
    # rms a sample, so rho to that over sqrt(M), 1.9e-13 loud, 4.5 times that at its
    # largest: 8e-6 at 1e7, but above the tolerance at 1e8 and 1e9.
    for prec in ("split_bf16", "fp32", "fft_fp32", "bf16") + (("split_fp16",) if loud == "1e7" else ()):
        rho = torch.zeros((K, L), dtype=torch.float32, device="cuda")
        outs, _, _ = run(ctx, bank, [x], fs, prec, rho_out=rho)
        err = np.abs(rho.cpu().numpy().astype(np.float64) - ref["rho"])
        assert err.max() <= TOL[prec], (prec, err.max(), np.unravel_index(err.argmax(), err.shape))
        check_maxima(outs[0], ref, ref["rho"], TOL[prec], prec)
        check_sigma(outs[0], ref, TOL[prec])
    bf.bf_bank_destroy(bank)


# block sums of 1024 samples: one thread each up to 256 of them, 16 a thread in
# rounds of 4096 beyond
@pytest.mark.parametrize("n", [256 * 1024, 256 * 1024 + 1, 4096 * 1024 - 5, 4096 * 1024 + 1, 2 * 4096 * 1024 + 1025])
def test_long_series_scan(ctx, n):
    """sigma = sqrt(mean rho^2) and the maxima of two short templates over
    series whose scan takes one round or several, quiet and loud by turns."""
    fs, M = 1024.0, 64
    spec = synth.grid_spec([synth.LINEAR], [synth.ASC, synth.DESC], [M / fs], 60.0, 480.0, 1, 1)
    bank = bf.bf_bank_create_grid(ctx, spec, fs, M / fs, bf.BF_BANK_FP32)
    p = oracle_params(spec)
    rng = np.random.default_rng(n)
    x = rng.standard_normal(n)
    x *= 10.0 ** rng.integers(-3, 4, n // 4096 + 1).repeat(4096)[:n]
    x[n // 2:n // 2 + 3000] = 0.0
    x = x.astype(np.float32)
    # rho in FP64: sliding products by FFT would lose the quiet stretches, so by the 64 shifts
    L = n - M + 1
    nu = np.zeros(L)
    H = [oracle.template(int(p["track"][k]), int(p["sense"][k]), p["f_lo"][k], p["f_hi"][k], p["D"][k], fs, M, 0)
         for k in range(2)]
    c = np.zeros((2, L))
    for m in range(M):
        w = x[m:m + L].astype(np.float64)
        nu += w * w
        for k in range(2):
            c[k] += H[k][m] * w
    rho = np.where(nu > 0, c / np.sqrt(np.where(nu > 0, nu, 1.0)), 0.0)
    outs, _, _ = run(ctx, bank, [x], fs, "fp32")
    a = np.abs(rho)
    np.testing.assert_allclose(outs[0]["max"], a.max(1), atol=TOL["fp32"])
    np.testing.assert_allclose(outs[0]["sigma"], np.sqrt((rho ** 2).mean(1)), atol=TOL["fp32"])
    for k in range(2):
        assert a[k, outs[0]["argmax"][k]] >= a[k].max() - 2 * TOL["fp32"]
    bf.bf_bank_destroy(bank)
