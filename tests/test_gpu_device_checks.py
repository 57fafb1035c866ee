"""Device functions that no call of the library shows by themselves, through
device_checks.cu: the inverse window norm over its whole range, the bounded
wait of the correlation kernels, and the control's rank step for buckets far more
crowded than uniform keys make them."""
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lines(tmp_path_factory):
    from paper_1802_01685_gb300 import build as b
    exe = str(tmp_path_factory.mktemp("checks") / "device_checks")
    cmd = [b._nvcc()] + b.ARCH + ["-O3", "-std=c++17", "-I", b.INCLUDE, "-I", b.CSRC,
                                  os.path.join(HERE, "device_checks.cu"), "-o", exe, "-lpthread"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stderr[-3000:]
    return [ln.split() for ln in r.stdout.splitlines()]


def test_inverse_norm_is_fp64s(lines):
    """The root and the division round once each, the library's form once: they
    are at most 3 units of 2^-53 apart (one Newton step from FP32 is 315), and
    then round to another FP32 value for 2^-27 of all energies at most: 2 of 2^28,
    taken four times."""
    (_, worst, wrong), = [a for a in lines if a[0] == "norms"]
    assert float(worst) <= 3.0 and int(wrong) <= 8, (worst, wrong)


def test_wait_is_bounded_in_time(lines):
    """It ends at its limit, by the clock and not by a count of tries, and soon
    once another wait of the block has run out (64 tries)."""
    (_, ns, ok, ns_abort, ok_abort), = [a for a in lines if a[0] == "wait"]
    assert int(ok) == 0 and 20_000_000 <= int(ns) < 500_000_000, ns
    assert int(ok_abort) == 0 and int(ns_abort) < 500_000_000, ns_abort


def test_crowded_buckets(lines):
    got = [a for a in lines if a[0] == "crowded_wrong"]
    assert len(got) == 9 and all(int(a[3]) == 0 for a in got), got
