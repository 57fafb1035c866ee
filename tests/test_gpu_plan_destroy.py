"""A plan taken down while its last run is on the GPU."""
import pytest

from paper_1802_01685_gb300 import bf, synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__
    __graft_entry__.build()
    h = bf.bf_init()
    yield h
    bf.bf_destroy(h)


def test_destroy_waits_for_the_run(ctx):
    """A run on a stream writes the plan's buffers, page-locked host memory
    among them, which go back for other results with the plan."""
    fs, T = 4096.0, 1.0
    spec = synth.grid_spec([synth.POWERLAW], [synth.ASC], [T], 40.0, 400.0, 64, 64)
    bank = bf.bf_bank_create_grid(ctx, spec, fs, T, bf.BF_BANK_SPLIT_BF16)
    x = torch.randn(262144, device="cuda")
    plan = bf.bf_plan_create(ctx, bank, [262144], fs, bf.make_opts())
    st = torch.cuda.Stream()
    torch.cuda.synchronize()
    bf.bf_plan_run(plan, [x], st.cuda_stream)           # about 12 ms
    bf.bf_plan_destroy(plan)
    done = st.query()
    st.synchronize()
    bf.bf_bank_destroy(bank)
    assert done
