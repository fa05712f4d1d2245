"""The identity behind the FP64 kernels' half list of helicities: with zero top width, flipping every helicity
conjugates a tree amplitude, up to a sign common to all colour orderings, so |M_h|^2 = |M_~h|^2 per event, colour
flow and (tests/test_gpu_sde.py) single diagram.  Checked on the oracle, which evaluates every helicity."""
import numpy as np
import pytest


@pytest.mark.parametrize("ng", [0, 1, 2, 3])
def test_oracle_flipped_helicities_have_equal_squares(orc, ng):
    nh = orc.nhel(ng)
    mom, _, _ = orc.events(ng, 40 + ng, 5 if ng < 3 else 2)
    for p in mom:
        mh, jamps = orc.me_hel(ng, p, want_jamps=True)
        # FP64 rounding of sums of at most ~1e4 terms, far below 1e-12 of the largest helicity
        assert np.max(np.abs(mh - mh[::-1])) <= 1e-12 * mh.max()
        a = np.abs(jamps) ** 2
        assert a.shape[0] == nh
        assert np.max(np.abs(a - a[::-1])) <= 1e-12 * a.max()
