"""A generated bank's first chunk is synthesised beside the series' preparation.
A call that fails between the two (the series does not fit the budget) gives
its ring back once the synthesis is done, and the calls after it equal the
stored bank's bit for bit, from one chunk to several, on the library's and on a
caller's stream."""
import numpy as np
import pytest

from paper_1802_01685_gb300 import bf, synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

FS, M = 2048.0, 2048


@pytest.mark.parametrize("prec", ["split_bf16", "split_fp16", "fp32"])
def test_failed_call_between_begin_and_launch(prec):
    import __graft_entry__
    __graft_entry__.build()
    spec = synth.grid_spec([synth.LINEAR], [synth.ASC, synth.DESC], [1.0], 20.0, 1000.0, 64, 64)      # 8192 templates
    storage = {"split_bf16": bf.BF_BANK_SPLIT_BF16, "split_fp16": bf.BF_BANK_SPLIT_FP16, "fp32": bf.BF_BANK_FP32}[prec]
    rng = np.random.default_rng(8)
    x = rng.standard_normal(9001).astype(np.float32)
    long = torch.zeros(8 << 20, device="cuda")              # 96 MB of prefix alone
    cfg = bf.bf_config_default()
    cfg.hbm_budget = 96 << 20
    small, full = bf.bf_init(cfg), bf.bf_init()
    try:
        gen = bf.bf_bank_create_grid(small, spec, FS, 1.0, bf.BF_BANK_GENERATED)
        ref = bf.bf_bank_create_grid(full, spec, FS, 1.0, storage)
        st = torch.cuda.Stream()
        for k_end, stream in ((8192, None), (3000, None), (128, None), (8192, st.cuda_stream)):
            with pytest.raises(bf.BFError) as e:
                bf.bf_correlate(small, gen, [long], FS, bf.make_opts(precision=prec, bank_end=k_end))
            assert e.value.status == bf.BF_ENOMEM
            a = bf.bf_correlate(small, gen, [x], FS, bf.make_opts(precision=prec, bank_end=k_end, stream=stream))
            st.synchronize()
            b = bf.bf_correlate(full, ref, [x], FS, bf.make_opts(precision=prec, bank_end=k_end))
            got, want = bf.bf_result_copy_to_host(a, 0), bf.bf_result_copy_to_host(b, 0)
            for key in ("max", "argmax", "sigma"):
                if key == "sigma":
                    np.testing.assert_allclose(got[key], want[key], rtol=1e-6)     # FP64 sums in arrival order
                else:
                    np.testing.assert_array_equal(got[key], want[key], err_msg=f"{prec} {k_end} {key}")
            bf.bf_result_destroy(a)
            bf.bf_result_destroy(b)
        bf.bf_bank_destroy(gen)
        bf.bf_bank_destroy(ref)
    finally:
        bf.bf_destroy(small)
        bf.bf_destroy(full)
