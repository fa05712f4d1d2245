"""The autotuner times only launch shapes that the context's kernels read, and keeps the shared FP64 items: the number of
kernels it launches is that of its warm-up and four calls for each such shape."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("proc,prec,wt,shapes", [
    ("ggtt", 0, 0.0, 1), ("ggttg", 0, 0.0, 2), ("ggttgg", 0, 0.0, 2), ("ggttg", 2, 0.0, 3), ("ggttg", 0, 1.5, 1),
    ("ggttg", 1, 1.5, 1)])
def test_only_shapes_that_differ_are_timed(proc, prec, wt, shapes, tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2210_11122_gb300 as mg
    from paper_2210_11122_gb300 import build
    build.build()
    n = 64
    with mg.Context(proc, wt=wt) as ctx:
        mom = torch.zeros(ctx.mom_count(n), dtype=torch.float64, device="cuda")
        me = torch.zeros(n, dtype=torch.float64, device="cuda")
        n0 = mg.kernel_launches()
        ctx.rambo(1, n, 1500.0, mom)
        ctx.hel_filter(mom, n)
        n1 = mg.kernel_launches()
        ctx.sigmakin(mom, n, me, prec)
        call = mg.kernel_launches() - n1
        before = ctx.launch_shape(prec)
        n2 = mg.kernel_launches()
        ctx.autotune(prec, nevt=n, cache_path=str(tmp_path / "shapes.txt"))
        assert mg.kernel_launches() - n2 == (n1 - n0) + 4 * shapes * call
        after = ctx.launch_shape(prec)
        if shapes == 1:
            assert after == before
        assert after[2] & 32 == before[2] & 32           # MG_LAUNCH_SHARED
