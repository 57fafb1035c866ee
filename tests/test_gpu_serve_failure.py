"""A kernel error in the serving loop.  Launches serve several requests and the
status word says not which, so one bounded wait that runs out on the serving
stream (nothing signals it; it ends at its limit) fails every request active
then, not only the first to finish; later requests and calls on the context are
served as ever, and a call's own failure leaves the served requests alone."""
import time

import numpy as np
import pytest

from paper_1802_01685_gb300 import bf, synth

pytestmark = pytest.mark.gpu

FS, T = 2048.0, 1.0


@pytest.fixture(scope="module")
def setup():
    import __graft_entry__
    __graft_entry__.build()
    ctx = bf.bf_init()
    spec = synth.grid_spec([synth.LINEAR, synth.POWERLAW], [synth.ASC, synth.DESC], [1.0, 0.5], 20.0, 1000.0, 16, 16)
    bank = bf.bf_bank_create_grid(ctx, spec, FS, T, bf.BF_BANK_SPLIT_BF16)      # 2048 templates
    yield ctx, bank
    bf.bf_bank_destroy(bank)
    bf.bf_destroy(ctx)


def submit_two(ctx, bank, prec):
    """Two requests of some 50 ms and more, both admitted."""
    rng = np.random.default_rng(3)
    x = rng.standard_normal(6 << 20).astype(np.float32)
    opts = bf.make_opts(precision=prec)
    tickets = [bf.bf_serve_submit(ctx, bank, x[:n], FS, opts) for n in (6 << 20, 4 << 20)]
    for _ in range(10000):
        if bf.bf_serve_stats_get(ctx).active == 2:
            return tickets
        time.sleep(1e-4)
    raise AssertionError("the requests were not active together")


@pytest.mark.parametrize("prec", ["split_bf16", "fft_fp32"])
def test_every_active_request_fails(setup, prec):
    ctx, bank = setup
    tickets = submit_two(ctx, bank, prec)
    bf.bf_selftest_serve(ctx, 1000)
    for t in tickets:
        with pytest.raises(bf.BFError) as e:
            bf.bf_serve_poll(ctx, t, 60_000_000)
        assert e.value.status == bf.BF_EDEVICE, t
    # and the loop goes on
    x = np.random.default_rng(4).standard_normal(9001).astype(np.float32)
    opts = bf.make_opts(precision=prec)
    st, res = bf.bf_serve_poll(ctx, bf.bf_serve_submit(ctx, bank, x, FS, opts), 60_000_000)
    assert st == bf.BF_OK
    ref = bf.bf_correlate(ctx, bank, [x], FS, opts)
    a, b = bf.bf_result_copy_to_host(res, 0), bf.bf_result_copy_to_host(ref, 0)
    for k in ("max", "argmax"):
        np.testing.assert_array_equal(a[k], b[k])
    bf.bf_result_destroy(res)
    bf.bf_result_destroy(ref)


def test_a_calls_failure_is_its_own(setup):
    ctx, bank = setup
    tickets = submit_two(ctx, bank, "split_bf16")
    with pytest.raises(bf.BFError) as e:
        bf.bf_selftest_wait(ctx, False, 20_000)
    assert e.value.status == bf.BF_EDEVICE
    for t in tickets:
        st, res = bf.bf_serve_poll(ctx, t, 60_000_000)
        assert st == bf.BF_OK
        bf.bf_result_destroy(res)


def test_limits(setup):
    ctx, bank = setup
    for limit in (0, 1_000_001):
        with pytest.raises(bf.BFError) as e:
            bf.bf_selftest_serve(ctx, limit)
        assert e.value.status == bf.BF_EINVAL
