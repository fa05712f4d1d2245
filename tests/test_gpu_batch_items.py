"""mg_sigmakin_batch with the FP64 items shared between combinations (the default launch shape): against the FP64 oracle
on its own momenta (1e-12 per event) and bit for bit against mg_sigmakin, over page edges, a partial helicity mask, jobs
with and without shared items in one batch, and jobs whose items exceed the 2 GiB that one launch holds."""
import os

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SQRTS = 1500.0
NTHREADS = os.cpu_count() or 1
SHARED, UNSHARED = 39, 7


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import oracle
    import paper_2210_11122_gb300 as mg
    from paper_2210_11122_gb300 import build
    build.build()
    oracle.build()
    return torch, mg, oracle


# (n_g, events, seed, helicity threshold, launch flags)
MIX = [(3, 13, 71, 1e-9, SHARED), (0, 1000, 72, 1e-9, SHARED), (1, 257, 73, 1e-9, SHARED), (2, 37, 74, 1e-9, SHARED),
       (1, 32, 75, 0.02, SHARED), (0, 33, 76, 1e-9, SHARED), (2, 129, 77, 0.01, SHARED), (3, 1, 78, 0.005, SHARED)]


@pytest.mark.parametrize("some_unshared", [False, True])
def test_shared_jobs_match_oracle_and_single_launches(env, some_unshared):
    torch, mg, orc = env
    ctxs, moms, mes, refs, partial = [], [], [], [], 0
    try:
        for i, (ng, n, seed, tau, flags) in enumerate(MIX):
            evs, _, _ = orc.events(ng, seed, n)
            mask, _ = orc.hel_mask(ng, evs, tau=tau, nthreads=NTHREADS)
            partial += ng > 0 and not np.array_equal(mask, orc.full_mask(ng))
            refs.append(orc.me_batch(ng, evs, mask=mask, nthreads=NTHREADS))
            c = mg.Context(ng, hel_warmup=1024, hel_tau=tau)
            c.set_launch_shape(mg.MG_FP64, 128, 0, UNSHARED if some_unshared and i % 3 == 2 else flags)
            ctxs.append(c)
            moms.append(torch.from_numpy(mg.to_aosoa(evs)).cuda())
            mes.append(torch.full((n + 1,), -1.0, dtype=torch.float64, device="cuda"))
        assert partial >= 2                                  # jobs on the helicity basis
        mg.sigmakin_batch([(c, m, job[1], me) for c, m, job, me in zip(ctxs, moms, MIX, mes)])
        for c in ctxs:
            assert c.check() == 0
        for (ng, n, _, tau, _), c, m, me, r in zip(MIX, ctxs, moms, mes, refs):
            g = me.cpu().numpy()
            assert g[n] == -1.0
            assert np.max(np.abs(g[:n] / r - 1)) <= 1e-12, (ng, n, tau)
            one = torch.zeros(n, dtype=torch.float64, device="cuda")
            c.sigmakin(m, n, one, mg.MG_FP64)
            assert np.array_equal(one.cpu().numpy(), g[:n]), (ng, n, tau)
    finally:
        for c in ctxs:
            c.close()


@pytest.mark.parametrize("jobs", [[(3, 7008)], [(2, 53696), (0, 100), (3, 6944)], [(3, 6976), (1, 65)]])
def test_jobs_over_the_items_bound(env, jobs):
    """6,944 gg -> t tbar g g g and 53,664 gg -> t tbar g g events fill 2 GiB of items: a larger job runs in chunks of
    its own launches, so a second batch call makes more launches than the persistent one alone, and none of it allocates."""
    torch, mg, orc = env
    ctxs = [mg.Context(p) for p, _ in jobs]
    try:
        moms = [torch.zeros(c.mom_count(n), dtype=torch.float64, device="cuda") for c, (_, n) in zip(ctxs, jobs)]
        mes = [torch.zeros(n, dtype=torch.float64, device="cuda") for _, n in jobs]
        want = []
        for c, m, (p, n) in zip(ctxs, moms, jobs):
            c.rambo(5 + p, n, SQRTS, m)
            me = torch.zeros(n, dtype=torch.float64, device="cuda")
            c.sigmakin(m, n, me, mg.MG_FP64)
            want.append(me)
        n0 = mg.kernel_launches()
        for c, m, (p, n), me in zip(ctxs, moms, jobs, want):
            c.sigmakin(m, n, me, mg.MG_FP64)
        single = mg.kernel_launches() - n0
        args = [(c, m, n, me) for c, m, (_, n), me in zip(ctxs, moms, jobs, mes)]
        mg.sigmakin_batch(args)
        for me, w in zip(mes, want):
            assert torch.equal(me, w)
            me.zero_()
        n0 = mg.kernel_launches()
        mg.diag_fail_alloc(1)
        mg.sigmakin_batch(args)
        mg.diag_fail_alloc(0)
        for me, w in zip(mes, want):
            assert torch.equal(me, w)
        # one persistent launch in place of the matrix-element launch of each job within the bound (none: no launch)
        small = sum(1 for p, n in jobs if n <= {0: 1 << 40, 1: 400000, 2: 53664, 3: 6944}[p])
        assert mg.kernel_launches() - n0 == single - small + (1 if small else 0)
    finally:
        mg.diag_fail_alloc(0)
        for c in ctxs:
            c.close()


def test_persistent_graph_with_a_job_over_the_bound(env):
    """The chunks of such a job are captured with the rest; contexts that have run nothing capture and replay."""
    torch, mg, orc = env
    sizes = [(3, 7008), (1, 65), (0, 33)]
    ctxs = []
    try:
        def graph(persistent):
            jobs = []
            for i, (p, n) in enumerate(sizes):
                c = mg.Context(p)
                ctxs.append(c)
                mom = torch.zeros(c.mom_count(n), dtype=torch.float64, device="cuda")
                me = torch.full((n,), -1.0, dtype=torch.float64, device="cuda")
                jobs.append((c, 60 + i, 0, n, SQRTS, mom, me, mg.MG_FP64))
            return mg.GraphBatch(jobs, persistent=persistent), jobs
        (ga, ja), (gb, jb) = graph(True), graph(False)
        for _ in range(2):
            ga.launch()
            gb.launch()
            torch.cuda.synchronize()
            for a, b in zip(ja, jb):
                assert torch.equal(a[6], b[6]) and bool((a[6] > 0).all())
                a[6].zero_()
                b[6].zero_()
        ga.close()
        gb.close()
    finally:
        for c in ctxs:
            c.close()
