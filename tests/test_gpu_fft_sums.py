"""What the FFT route's epilogue reduces: a NaN of an overflowing transform
reaches the maximum, and the sum of rho^2 rounds in FP32 over chains of 32 terms
only, those being added as pairs of FP32 values and then in FP64."""
import numpy as np
import pytest

from paper_1802_01685_gb300 import bf, synth

from parity import run

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

FS, M = 4096.0, 1024


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__
    __graft_entry__.build()
    h = bf.bf_init()
    yield h
    bf.bf_destroy(h)


@pytest.fixture(scope="module", params=[False, True])
def bank(ctx, request):
    spec = synth.grid_spec([synth.LINEAR, synth.POWERLAW], [synth.ASC, synth.DESC], [M / FS], 40.0, 1500.0, 16, 32)
    b = bf.bf_bank_create_grid(ctx, spec, FS, M / FS,
                               bf.BF_BANK_FP32 | (bf.BF_BANK_QUADRATURE if request.param else 0))
    yield b, request.param
    bf.bf_bank_destroy(b)


@pytest.mark.parametrize("n", [9000, 60000])
def test_large_finite_samples(ctx, bank, n):
    """Samples are finite float32 of any size.  Where the transform holds them
    the outputs equal those of the same series at 1 (a power of two apart, so
    bit for bit; a quadrature bank squares them, which ends sooner); past that they
    are NaN, not a maximum of 0 at no lag, in whichever segment the overflow lies."""
    b, quad = bank
    rng = np.random.default_rng(n)
    x = rng.standard_normal(n).astype(np.float32)
    one = run(ctx, b, [x], FS, "fft_fp32")[0][0]
    big = run(ctx, b, [x * np.float32(2.0 ** (40 if quad else 90))], FS, "fft_fp32")[0][0]
    np.testing.assert_array_equal(big["max"], one["max"])
    np.testing.assert_array_equal(big["argmax"], one["argmax"])
    L = n - M + 1
    for where in (slice(0, n), slice(0, 2000), slice(n - 2000, n)):
        y = x.copy()
        y[where] *= np.float32(1e37)
        out = run(ctx, b, [y], FS, "fft_fp32")[0][0]
        assert np.isnan(out["max"]).all(), where
        assert np.isnan(out["sigma"]).all(), where
        assert ((out["argmax"] >= 0) & (out["argmax"] < L)).all(), where


def test_sigma_is_the_rounded_sum(ctx, bank):
    """One segment: sigma against the FP64 sum of the dense rho^2.  In FP32
    only chains of 32 terms (16 with a quadrature bank) are added, whose rounding
    shows in about 1-2 % of the sigmas (an emulation of the kernel's order:
    0.009 to 0.021 over 300 to 12,289 lags); with the lanes' tree in FP32 too it
    was 7-13 %."""
    b, K = bank[0], 2048
    rng = np.random.default_rng(5)
    wrong = total = 0
    for n in (M + 2000, M + 7000):
        x = rng.standard_normal(n).astype(np.float32)
        rho = torch.zeros((K, n - M + 1), dtype=torch.float32, device="cuda")
        out = run(ctx, b, [x], FS, "fft_fp32", rho_out=rho)[0][0]
        want = torch.sqrt((rho.double() ** 2).mean(1)).float().cpu().numpy()
        np.testing.assert_allclose(out["sigma"], want, rtol=2.5e-7)
        wrong += int((out["sigma"] != want).sum())
        total += K
    assert wrong <= 0.04 * total, wrong / total
