"""The host copy that the finalize kernels write beside a result.  What
bf_result_copy_to_host gives from it equals, bit for bit, the device arrays
(read through bf_result_copy_to_host_async), for results below and above the
size up to which outputs are mirrored (4 MiB), and after plan runs in either
mode: a run on a stream must not leave the run before in the host copy."""
import numpy as np
import pytest

from paper_1802_01685_gb300 import bf, synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

FS, T, M = 1024.0, 0.0625, 64


@pytest.fixture(scope="module")
def setup():
    import __graft_entry__
    __graft_entry__.build()
    ctx = bf.bf_init()
    spec = synth.grid_spec([synth.LINEAR], [synth.ASC, synth.DESC], [T], 60.0, 500.0, 32, 64)      # 4096 templates
    bank = bf.bf_bank_create_grid(ctx, spec, FS, T, bf.BF_BANK_SPLIT_BF16)
    yield ctx, bank
    bf.bf_bank_destroy(bank)
    bf.bf_destroy(ctx)


def device_arrays(res, s, K, hist):
    t = dict(max=torch.empty(K, dtype=torch.float32), argmax=torch.empty(K, dtype=torch.int32),
             sigma=torch.empty(K, dtype=torch.float32))
    if hist:
        t["hist"] = torch.empty(1024, dtype=torch.int32)
    t = {k: v.pin_memory() for k, v in t.items()}
    out = {k: v.numpy().view(np.uint32) if k == "hist" else v.numpy() for k, v in t.items()}
    st = torch.cuda.Stream()
    bf.bf_result_copy_to_host_async(res, s, out, st.cuda_stream, want_hist=hist)
    st.synchronize()
    return out


def check(res, n, K, hist):
    for s in range(n):
        a, b = bf.bf_result_copy_to_host(res, s, want_hist=hist), device_arrays(res, s, K, hist)
        for k, v in b.items():
            np.testing.assert_array_equal(a[k], v, err_msg=f"series {s} {k}")


@pytest.mark.parametrize("n,k_end,hist", [(1, 1, True), (1, 4096, False), (3, 1000, True), (80, 4096, True),
                                          (90, 4096, False)])           # 3.9 and 4.4 MB
def test_host_copy_equals_device_arrays(setup, n, k_end, hist):
    ctx, bank = setup
    rng = np.random.default_rng(n + k_end)
    xs = [rng.standard_normal(M + 3 * i + 1).astype(np.float32) for i in range(n)]
    res = bf.bf_correlate(ctx, bank, xs, FS, bf.make_opts(bank_end=k_end, want_hist=hist))
    check(res, n, k_end, hist)
    vm = np.stack([bf.bf_result_copy_to_host(res, s, want_hist=False)["max"] for s in range(n)])
    np.testing.assert_allclose(bf.bf_result_copy_mean_max(res), vm.astype(np.float64).mean(0), rtol=1e-6)
    assert bf.bf_result_info_get(res).n_candidates >= 0
    bf.bf_result_destroy(res)


def test_plan_runs_in_either_mode(setup):
    ctx, bank = setup
    plan = bf.bf_plan_create(ctx, bank, [500, 300], FS, bf.make_opts())
    try:
        st = torch.cuda.Stream()
        seen = []
        for run in range(4):
            rng = np.random.default_rng(run)
            xs = [torch.from_numpy(rng.standard_normal(k).astype(np.float32)).cuda() for k in (500, 300)]
            res = bf.bf_plan_run(plan, xs, st.cuda_stream if run % 2 else None)
            st.synchronize()
            check(res, 2, 4096, True)
            seen.append(bf.bf_result_copy_to_host(res, 0)["max"])
        assert not any(np.array_equal(seen[i], seen[i + 1]) for i in range(3))
    finally:
        bf.bf_plan_destroy(plan)
