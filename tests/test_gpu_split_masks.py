"""FP64 entry points under masks that keep one helicity of some flipped pairs (weights 0, 1 and 2 of the pair) against the
oracle with the same mask: matrix elements, LHE choices, mg_sigmakin_noalloc, channel weights, the tensor-core colour sum and
the persistent batch.  The two helicities of a pair have the same ratio up to the filter's FP32 rounding, so a threshold
at a pair's exact ratio splits some of them (from three gluons; with two the FP32 sums of a pair are equal); the mask the
filter then finds is taken as given.

Bounds: 1e-12 of the event's full matrix element (every helicity: what FP64 rounding is relative to), 1e-6 for the
tensor-core colour sum, 1e-12 of the largest weight; a choice may differ from the oracle's only within 1e-12 of a boundary."""
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
    import oracle.lhe as olhe
    import oracle.sde as osde
    import paper_2210_11122_gb300 as mg
    from paper_2210_11122_gb300 import build
    build.build()
    oracle.build()
    return torch, mg, oracle, olhe, osde


def bits(mask, nhel):
    return np.array([(int(mask[h >> 5]) >> (h & 31)) & 1 for h in range(nhel)])


def near_boundary(weights, r):
    tot = float(np.sum(weights))
    return bool(np.any(np.abs(np.cumsum(weights) - r * tot) <= 1e-12 * tot))


@pytest.mark.parametrize("ng,n", [(1, 70), (2, 33), (3, 5)])
def test_fp64_entry_points_under_a_split_mask(env, ng, n):
    torch, mg, orc, olhe, osde = env
    evs, _, _ = orc.events(ng, 500 + ng, n)
    nhel = orc.nhel(ng)
    _, ratio = orc.hel_mask(ng, evs, nthreads=NTHREADS)
    mom = torch.from_numpy(mg.to_aosoa(evs)).cuda()
    full = orc.me_batch(ng, evs, nthreads=NTHREADS)
    found = 0
    r = np.unique(np.round(np.log(ratio[ratio > 1e-20]), 9))
    for tau in np.exp(r[len(r) // 4:]):                     # (the smaller ratios keep all but a few helicities)
        with mg.Context(ng, hel_warmup=n, hel_tau=float(tau)) as ctx:
            ctx.hel_filter(mom, n)
            mask, ngood = ctx.hel_mask()
            b = bits(mask, nhel)
            if ngood == 0 or np.array_equal(b, b[::-1]):
                continue
            found += 1
            ref = orc.me_batch(ng, evs, mask=mask, nthreads=NTHREADS)
            me = torch.zeros(n, dtype=torch.float64, device="cuda")

            def check(got, bound=1e-12):
                assert np.max(np.abs(got.cpu().numpy() - ref) / full) <= bound
            for flags in (39, 7):
                ctx.set_launch_shape(mg.MG_FP64, 128, 0, flags)
                ctx.sigmakin(mom, n, me, mg.MG_FP64)
                check(me)
                ctx.set_launch_shape(mg.MG_FP64_TCCOLOR, 128, 0, flags)
                ctx.sigmakin(mom, n, me, mg.MG_FP64_TCCOLOR)
                check(me, 1e-6)
            ctx.set_launch_shape(mg.MG_FP64, 128, 0, 39)
            ctx.sigmakin(mom, n, me, mg.MG_FP64)
            one = me.clone()
            mg.sigmakin_batch([(ctx, mom, n, me)])
            assert torch.equal(me, one)
            ctx.sigmakin_noalloc(mom, n, me)
            check(me)
            rng = np.random.default_rng(900 + found)
            rh, rc = rng.random(n), rng.random(n)
            hel = torch.full((n,), -1, dtype=torch.int32, device="cuda")
            col = torch.full((n,), -1, dtype=torch.int32, device="cuda")
            ctx.sigmakin_lhe(mom, n, me, torch.from_numpy(rh).cuda(), torch.from_numpy(rc).cuda(), hel, col)
            check(me)
            dias = osde.diagrams(ng)
            pos = {osde.key(d): i for i, d in enumerate(dias)}
            order = [pos[k] for k in mg.sde_channels(ng)]
            w = torch.zeros(len(order) * n, dtype=torch.float64, device="cuda")
            ctx.sde_weights(mom, n, w)
            w = w.cpu().numpy().reshape(len(order), n)
        for e in range(n):
            _, rhel, rcol, _, det = olhe.event(ng, evs[e], mask, r_hel=rh[e], r_col=rc[e])
            assert b[int(hel[e])]
            assert int(hel[e]) == rhel or near_boundary([det["mh"][h] for h in det["good"]], rh[e])
            assert int(col[e]) == rcol or near_boundary(det["w"], rc[e])
        for e in (0, n - 1):
            refw = osde.weights(ng, evs[e], mask, dias=dias)[order]
            assert np.max(np.abs(w[:, e] - refw)) <= 1e-12 * refw.max()
        if found == 2:
            break
    assert found > 0
