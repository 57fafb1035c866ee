"""Per-device set-up (csrc/device_once.h) on the CPU, with a stand-in for
cudaGetDevice: it runs once on each device, again where it failed, and once only
when many threads come at the same time.  Both users of it go through it."""
import os
import subprocess
import textwrap

from paper_1802_01685_gb300 import build as b

_MAIN = textwrap.dedent("""
    #include <atomic>
    #include <cstdio>
    #include <thread>
    #include "device_once.h"
    static thread_local int current = 0;
    extern "C" cudaError_t cudaGetDevice(int* d) { *d = current; return cudaSuccess; }
    int main()
    {
        bfi::DeviceOnce once;
        std::atomic<int> ran[3] = {};
        bool fail = true;
        auto set = [&] { ++ran[current]; return current == 2 && fail ? cudaErrorInvalidValue : cudaSuccess; };
        std::thread t[16];
        for (int i = 0; i < 16; ++i)
            t[i] = std::thread([&, i] {
                for (int n = 0; n < 1000; ++n) {
                    current = (i + n) & 1;
                    if (once.run(set) != cudaSuccess) ++ran[2];
                }
            });
        for (auto& x : t) x.join();
        std::printf("%d %d %d", (int)ran[0], (int)ran[1], (int)ran[2]);
        current = 2;
        const cudaError_t a = once.run(set);
        fail = false;
        const cudaError_t c = once.run(set), d = once.run(set);
        std::printf(" %d %d %d %d\\n", a != cudaSuccess, c, d, (int)ran[2]);
    }
""")


def test_once_on_each_device(tmp_path):
    src, exe = tmp_path / "m.cpp", tmp_path / "m"
    src.write_text(_MAIN)
    cuda = os.path.join(os.path.dirname(os.path.dirname(b._nvcc())), "include")
    cmd = ["g++", "-std=c++17", "-O1", "-I", b.CSRC, "-I", cuda, str(src), "-o", str(exe), "-lpthread"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.stdout.split() == "1 1 0 1 0 0 2".split()


def test_every_shared_memory_opt_in_is_per_device():
    for f in ("corr_tc.cu", "corr_fft.cu"):
        text = open(os.path.join(b.CSRC, f)).read()
        assert "static DeviceOnce once;" in text and "static bool" not in text, f
