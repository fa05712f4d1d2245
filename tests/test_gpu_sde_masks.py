"""Channel weights under a partial helicity mask (a threshold in the widest gap of the oracle's per-helicity maximum
ratios), every process, against the oracle's weights for that mask: 1e-12 of the largest weight, the bound of the other
tests of the weights.  The helicity kernels and those of the linear polarisations end in one normalising launch."""
import os

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ng,n", [(0, 33), (1, 1), (1, 65), (2, 33), (3, 5)])
def test_weights_under_a_partial_mask(ng, n):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import oracle as orc
    from oracle import sde
    import paper_2210_11122_gb300 as mg
    from paper_2210_11122_gb300 import build
    build.build()
    orc.build()
    evs, _, _ = orc.events(ng, 177 + ng, n)
    _, ratio = orc.hel_mask(ng, evs, nthreads=os.cpu_count() or 1)
    r = np.sort(ratio[ratio > 1e-20])
    mid = len(r) // 2
    k = max(range(mid - len(r) // 4, mid + len(r) // 4), key=lambda i: r[i + 1] / r[i])
    tau = float(np.sqrt(r[k] * r[k + 1]))
    mask, _ = orc.hel_mask(ng, evs, tau=tau)
    ngood = sum(bin(int(w)).count("1") for w in mask)
    assert 0 < ngood < orc.nhel(ng)
    dias = sde.diagrams(ng)
    pos = {sde.key(d): i for i, d in enumerate(dias)}
    order = [pos[key] for key in mg.sde_channels(ng)]
    with mg.Context(ng, hel_tau=tau, hel_warmup=n) as ctx:
        mom = torch.from_numpy(mg.to_aosoa(evs)).cuda()
        ctx.hel_filter(mom, n)
        assert np.array_equal(ctx.hel_mask()[0], mask)
        w = torch.zeros(len(order) * n, dtype=torch.float64, device="cuda")
        ctx.sde_weights(mom, n, w)          # (first call: uploads the tables)
        n0 = mg.kernel_launches()
        ctx.sde_weights(mom, n, w)
        # record, helicities, normalisation; from three gluons on the K - 1 passes and the channels of the other basis
        assert mg.kernel_launches() - n0 == (3 if ng == 0 else 3 + (ng + 1) + 1)
        got = w.cpu().numpy().reshape(len(order), n)
    for e in sorted({0, n // 2, n - 1}):
        ref = sde.weights(ng, evs[e], mask, dias=dias)[order]
        assert np.max(np.abs(got[:, e] - ref)) <= 1e-12 * ref.max()
