"""Scratch grows with the largest batch only: once a context has run a batch, a smaller one allocates nothing, whatever
chunks the two are cut into, so it can also be captured into a CUDA graph.  Sizes on both sides of the chunk limits of
the FP64 items (gg -> t tbar g g g: 6,944 events, with the amplitudes 4,960; gg -> t tbar g g: 53,664)."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2210_11122_gb300 as mg
    from paper_2210_11122_gb300 import build
    build.build()
    yield torch, mg
    mg.diag_fail_alloc(0)


@pytest.mark.parametrize("proc,large,small,kind", [
    ("ggttggg", 8192, 6000, "fp64"), ("ggttggg", 8192, 4097, "fp64"), ("ggttgg", 60000, 50000, "fp64"),
    ("ggttggg", 5400, 4960, "tc"), ("ggttggg", 5400, 4960, "lhe")])
def test_smaller_batch_allocates_nothing(env, proc, large, small, kind):
    torch, mg = env
    with mg.Context(proc) as ctx:
        mom = torch.zeros(ctx.mom_count(large), dtype=torch.float64, device="cuda")
        me = torch.zeros(large, dtype=torch.float64, device="cuda")
        ctx.rambo(9, large, 1500.0, mom)

        def call(n, stream=None):
            if kind == "lhe":
                ctx.sigmakin_lhe(mom, n, me, stream=stream)
            else:
                ctx.sigmakin(mom, n, me, mg.MG_FP64 if kind == "fp64" else mg.MG_FP64_TCCOLOR, stream=stream)
        call(large)
        torch.cuda.synchronize()
        ref = me[:small].clone()
        me.zero_()
        torch.cuda.synchronize()
        mg.diag_fail_alloc(1)                 # the next allocation of the library fails
        call(small)
        mg.diag_fail_alloc(0)
        torch.cuda.synchronize()
        assert torch.equal(me[:small], ref)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            call(small, torch.cuda.current_stream())
        me.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(me[:small], ref)
