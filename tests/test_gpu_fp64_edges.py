"""The FP64 paths at the edges of their 32-event pages, against the FP64 oracle on its own momenta (1e-12 per event, the
bound of every FP64 parity test): matrix elements with and without the shared items, the tensor-core colour sum and the
LHE matrix elements; and the channel weights with every helicity good and with a partial mask (both code paths)."""
import os

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
NTHREADS = os.cpu_count() or 1


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import oracle
    import paper_2210_11122_gb300 as mg
    from paper_2210_11122_gb300 import build
    build.build()
    oracle.build()
    return torch, mg, oracle


@pytest.mark.parametrize("ng", [0, 1, 2, 3])
@pytest.mark.parametrize("n", [1, 31, 32, 33, 65])
def test_fp64_paths_at_page_edges(env, ng, n):
    torch, mg, orc = env
    if ng == 3 and n == 65:
        n = 34
    evs, _, _ = orc.events(ng, 300 + n, n)
    mask, _ = orc.hel_mask(ng, evs, nthreads=NTHREADS)
    ref = orc.me_batch(ng, evs, mask=mask, nthreads=NTHREADS)
    with mg.Context(ng) as ctx:
        mom = torch.from_numpy(mg.to_aosoa(evs)).cuda()
        ctx.hel_filter(mom, n)
        got = {}
        for flags in (39, 7):
            for prec in (mg.MG_FP64, mg.MG_FP64_TCCOLOR):
                ctx.set_launch_shape(prec, 128, 0, flags)
                me = torch.full((n + 1,), -1.0, dtype=torch.float64, device="cuda")
                ctx.sigmakin(mom, n, me, prec)
                out = me.cpu().numpy()
                assert out[n] == -1.0                     # nothing past the batch
                # the tensor-core colour sum takes FP32 jamps split into FP16 pairs: 1e-5 per event, its documented bound
                assert np.max(np.abs(out[:n] / ref - 1)) <= (1e-12 if prec == mg.MG_FP64 else 1e-5), (flags, prec)
                got[prec, flags] = out[:n]
            me = torch.zeros(n, dtype=torch.float64, device="cuda")
            ctx.sigmakin_lhe(mom, n, me)
            assert np.max(np.abs(me.cpu().numpy() / ref - 1)) <= 1e-12
        assert np.array_equal(got[mg.MG_FP64, 39], got[mg.MG_FP64, 7])
        assert np.array_equal(got[mg.MG_FP64_TCCOLOR, 39], got[mg.MG_FP64_TCCOLOR, 7])


@pytest.mark.parametrize("ng", [1, 2])
def test_channel_weights_of_both_paths(env, ng):
    """A threshold just above the smallest maximum ratio drops helicities, which takes the helicity kernels; the weights
    are the oracle's for that mask, as they are with every helicity good (linear polarisations)."""
    torch, mg, orc = env
    from oracle import sde
    n = 33
    evs, _, _ = orc.events(ng, 77 + ng, n)
    full, ratio = orc.hel_mask(ng, evs, nthreads=NTHREADS)
    ratio = np.sort(np.asarray(ratio)[: orc.nhel(ng)])
    gap = np.argmax(ratio[1:] / ratio[:-1])               # the widest gap between maximum ratios
    dias = sde.diagrams(ng)
    pos = {sde.key(d): i for i, d in enumerate(dias)}
    order = [pos[k] for k in mg.sde_channels(ng)]
    for tau in (1e-9, float(np.sqrt(ratio[gap] * ratio[gap + 1]))):
        mask, _ = orc.hel_mask(ng, evs, tau=tau, nthreads=NTHREADS)
        with mg.Context(ng, hel_tau=tau) as ctx:
            mom = torch.from_numpy(mg.to_aosoa(evs)).cuda()
            ctx.hel_filter(mom, n)
            assert np.array_equal(ctx.hel_mask()[0], mask)
            w = torch.zeros(len(order) * n, dtype=torch.float64, device="cuda")
            ctx.sde_weights(mom, n, w)
            got = w.cpu().numpy().reshape(len(order), n)
        for e in (0, 31, 32):
            ref = sde.weights(ng, evs[e], mask, dias=dias)[order]
            assert np.max(np.abs(got[:, e] - ref)) <= 1e-12 * ref.max()


@pytest.mark.parametrize("precision", [0, 2])
def test_graph_of_fresh_contexts(env, precision):
    """mg_graph_create reserves every scratch buffer of the FP64 modes before it captures: contexts that have run nothing
    capture and replay, and give the bits of the same steps called one by one."""
    torch, mg, orc = env
    sizes = {0: 300, 1: 200, 2: 97, 3: 40}
    ctxs = {p: mg.Context(p) for p in sizes}
    bufs = {p: (torch.zeros(ctxs[p].mom_count(n), dtype=torch.float64, device="cuda"),
                torch.zeros(n, dtype=torch.float64, device="cuda")) for p, n in sizes.items()}
    g = mg.GraphBatch([(ctxs[p], 11 + p, 0, n, 1500.0, bufs[p][0], bufs[p][1], precision) for p, n in sizes.items()])
    live = mg.live_allocs()
    g.launch()
    torch.cuda.synchronize()
    assert mg.live_allocs() == live
    for p, n in sizes.items():
        with mg.Context(p) as c:
            mom = torch.zeros(c.mom_count(n), dtype=torch.float64, device="cuda")
            me = torch.zeros(n, dtype=torch.float64, device="cuda")
            c.rambo(11 + p, n, 1500.0, mom)
            c.hel_filter(mom, n)
            c.sigmakin(mom, n, me, precision)
            assert torch.equal(me, bufs[p][1]), p
    g.close()
    for c in ctxs.values():
        c.close()
