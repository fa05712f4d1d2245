"""mg_sigmakin_host splits large batches into chunks of at least 131,072 events whose copies overlap the matrix elements
of other chunks: the results are those of one device-buffer call bit for bit, over two, three and four chunks with a
ragged last one, and the launches show that the batch was split."""
import pytest

pytestmark = pytest.mark.gpu
CHUNK = 131072


@pytest.mark.parametrize("proc,nevt,prec,chunks", [
    ("ggtt", 2 * CHUNK - 1, 0, 1), ("ggtt", 2 * CHUNK, 1, 2), ("ggtt", 2 * CHUNK + 17, 0, 2), ("ggtt", 4 * CHUNK + 96, 1, 4),
    ("ggttg", 3 * CHUNK + 33, 3, 3), ("ggttg", 6 * CHUNK + 1, 1, 4), ("ggttg", 2 * CHUNK + 31, 0, 2)])
def test_host_chunks_equal_one_device_call(proc, nevt, prec, chunks):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2210_11122_gb300 as mg
    from paper_2210_11122_gb300 import build
    build.build()
    with mg.Context(proc) as ctx:
        mom = torch.zeros(ctx.mom_count(nevt), dtype=torch.float64, device="cuda")
        ctx.rambo(5, nevt, 1500.0, mom)
        ctx.hel_filter(mom, 1024)
        me = torch.zeros(nevt, dtype=torch.float64, device="cuda")
        n0 = mg.kernel_launches()
        ctx.sigmakin(mom, nevt, me, prec)
        one = mg.kernel_launches() - n0
        host_mom = mom.cpu().pin_memory()
        host_me = torch.full((nevt,), -1.0, dtype=torch.float64).pin_memory()
        n0 = mg.kernel_launches()
        ctx.sigmakin_host(host_mom, nevt, host_me, prec)
        # (FP64 gg -> t tbar g runs its own chunks of at most 2 GiB of items: as many launches or more per call)
        split = mg.kernel_launches() - n0
        assert split == chunks * one if proc == "ggtt" else split >= chunks
        assert torch.equal(me.cpu(), host_me)
