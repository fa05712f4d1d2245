"""Rounding error of the phase-space weights (mg_rambo) against the same formulas in extended precision on the same
uniforms.  The boost's velocity and the weight's factors are quotients; formed as products with a rounded reciprocal they
cost fewer instructions and the weights lose a tenth of their accuracy."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
SQRTS, MT = 1500.0, 173.0
LD = np.longdouble


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    if np.finfo(LD).eps > 1e-18:
        pytest.skip("no extended precision on the host")
    import paper_2210_11122_gb300 as mg
    from paper_2210_11122_gb300 import build
    build.build()
    return torch, mg


def weights(u):
    """Phase-space weights of massive RAMBO for uniforms u[n, nf, 4], tops first (extended precision)."""
    n, nf = u.shape[:2]
    pi = LD("3.14159265358979323846264338327950288")
    c = 2 * u[..., 0] - 1
    s, phi, q0 = np.sqrt(1 - c * c), 2 * pi * u[..., 1], -np.log(u[..., 2] * u[..., 3])
    q = np.stack([q0, q0 * s * np.cos(phi), q0 * s * np.sin(phi), q0 * c], -1)
    Q = q.sum(1)
    M = np.sqrt(Q[:, 0] ** 2 - (Q[:, 1:] ** 2).sum(1))
    b, gam = -Q[:, 1:] / M[:, None], Q[:, 0] / M
    e0 = LD(SQRTS) / M[:, None] * (gam[:, None] * q[..., 0] + (b[:, None] * q[..., 1:]).sum(-1))
    m2 = np.zeros(nf, LD)
    m2[:2] = LD(MT) ** 2
    xi = np.full((n, 1), np.sqrt(1 - (2 * LD(MT) / LD(SQRTS)) ** 2))
    for _ in range(12):
        e = np.sqrt(m2 + (xi * e0) ** 2)
        xi = xi - (e.sum(1, keepdims=True) - LD(SQRTS)) / (xi * e0 * e0 / e).sum(1, keepdims=True)
    e, v = np.sqrt(m2 + (xi * e0) ** 2), xi * e0
    w0 = ((2 * pi) ** (4 - 3 * nf) * (pi / 2) ** (nf - 1) * LD(SQRTS) ** (2 * nf - 4)
          / (math.factorial(nf - 1) * math.factorial(nf - 2)))
    return w0 * xi[:, 0] ** (2 * nf - 3) * (v / e).prod(1) * LD(SQRTS) / (v * v / e).sum(1)


# medians of the relative error, divisions / reciprocals: 5.73e-16 / 6.28e-16 (one gluon), 7.79e-16 / 8.82e-16 (two);
# the bounds are the midpoints
@pytest.mark.parametrize("ng,n,bound", [(1, 8192, 6.0e-16), (2, 2048, 8.3e-16)])
def test_weights_keep_the_accuracy_of_divisions(env, ng, n, bound):
    torch, mg = env
    seed, nf = 11 + ng, ng + 2
    with mg.Context(ng) as ctx:
        mom = torch.zeros(ctx.mom_count(n), dtype=torch.float64, device="cuda")
        wgt = torch.zeros(n, dtype=torch.float64, device="cuda")
        ctx.rambo(seed, n, SQRTS, mom, wgt)
        words = torch.zeros(4 * n * nf, dtype=torch.int32, device="cuda")
        mg.philox(seed, n, nf, words)
        torch.cuda.synchronize()
    x = words.cpu().numpy().view(np.uint32).reshape(n, nf, 4)
    ref = weights((x.astype(LD) + LD(0.5)) * LD(2) ** -32)
    err = np.abs(np.asarray(wgt.cpu().numpy() / ref - 1, np.float64))
    assert np.median(err) <= bound, np.median(err)
    assert err.max() <= 1e-11
