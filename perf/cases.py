"""The engine's work as its users have it done, for timing and for comparing outputs.

Every case is one pass through the public entry points of paper_2210_11122_gb300: matrix elements of
given momenta in the precision modes (Context.sigmakin), the whole standalone step from a seed
(rambo + hel_filter + sigmakin), the host-buffer call (sigmakin_host), and the event-level epilogues
(sigmakin_lhe, sde_weights).  Contexts keep their default launch shapes, as in the README's example.
Momenta are flat massive phase space at sqrt(s) = 1500 GeV, made here with torch from the seed.

exact() evaluates the same outputs with plain torch in float64 / complex128: colour-ordered currents
of every gluon sequence, every helicity, the colour matrix from explicit Gell-Mann matrices.
"""
import itertools
import math

import numpy as np
import torch

import paper_2210_11122_gb300 as mg

SQRTS, MT, ALPHAS = 1500.0, 173.0, 0.118
NG = {"ggtt": 0, "ggttg": 1, "ggttgg": 2, "ggttggg": 3}
MODES = {"fp64": mg.MG_FP64, "fp32": mg.MG_FP32_AMP, "tc": mg.MG_FP64_TCCOLOR, "mixed": mg.MG_MIXED}


# ------------------------------------------------------------------------------------------
# the cases
# ------------------------------------------------------------------------------------------
def _case(kind, process, mode, nevt):
    return {"kind": kind, "process": process, "mode": mode, "nevt": int(nevt)}


def listed():
    def named(name, *a):
        return dict(_case(*a), name=name)

    return [
        # the smallest request of the serving trace: launch latency
        named("me_ggtt_fp64_32", "me", "ggtt", "fp64", 32),
        # the standalone step of the smallest process at its workload size: several short kernels
        named("step_ggtt_fp64_16384", "step", "ggtt", "fp64", 16384),
        # the benchmark's headline process at its workload size, in FP64 and with FP32 amplitudes
        named("me_ggttg_fp64_524288", "me", "ggttg", "fp64", 524288),
        named("me_ggttg_fp32_524288", "me", "ggttg", "fp32", 524288),
        # the paper's process: a ragged mid-size FP64 request, and the FP32 workload
        named("me_ggttgg_fp64_10007", "me", "ggttgg", "fp64", 10007),
        named("me_ggttgg_fp32_262144", "me", "ggttgg", "fp32", 262144),
        # five gluons: FP64, FP64 with the tensor-core colour sum (small odd batch), mixed at workload size
        named("me_ggttggg_fp64_8192", "me", "ggttggg", "fp64", 8192),
        named("me_ggttggg_tc_2049", "me", "ggttggg", "tc", 2049),
        named("me_ggttggg_mixed_65536", "me", "ggttggg", "mixed", 65536),
        # a generator with its momenta in host memory: copies in and out inside the call (the benchmark's
        # end-to-end form)
        named("host_ggttg_fp64_131073", "host", "ggttg", "fp64", 131073),
        # event-level epilogues: helicity and colour choices with the running coupling; channel weights
        named("lhe_ggttgg_32768", "lhe", "ggttgg", "fp64", 32768),
        named("sde_ggttg_65536", "sde", "ggttg", "fp64", 65536),
    ]


# the largest batch drawn of each kind, process by process (no more work than the largest listed case)
_CAP64 = {"ggtt": 524288, "ggttg": 524288, "ggttgg": 65536, "ggttggg": 8192}
_CAP32 = {"ggtt": 524288, "ggttg": 524288, "ggttgg": 262144, "ggttggg": 65536}
_CAPS = {"lhe": {"ggtt": 262144, "ggttg": 262144, "ggttgg": 65536, "ggttggg": 4096},
         "sde": {"ggttg": 131072, "ggttgg": 32768}}


def draw(rng):
    kind = rng.choices(["me", "step", "host", "lhe", "sde"], [6, 2, 1, 2, 1])[0]
    if kind in _CAPS:
        caps, mode = _CAPS[kind], "fp64"
    else:
        mode = rng.choice(list(MODES))
        caps = _CAP64 if mode in ("fp64", "tc") else _CAP32
    process = rng.choice(sorted(caps))
    nevt = int(round(math.exp(rng.uniform(math.log(16), math.log(caps[process])))))
    return _case(kind, process, mode, nevt)


# ------------------------------------------------------------------------------------------
# inputs
# ------------------------------------------------------------------------------------------
def _device():
    return torch.device("cuda") if torch.cuda.is_available() else torch.device("cpu")


def _rambo(u, sqrts=SQRTS, mt=MT):
    """Massive RAMBO (Kleiss, Stirling, Ellis): uniforms u[nevt, nf, 4] -> momenta [nevt, nf + 2, 4]
    (g1, g2, t, tbar, g3, ...) and phase-space weights."""
    nf = u.shape[1]
    c = 2.0 * u[..., 0] - 1.0
    s = 2.0 * torch.sqrt(u[..., 0] * (1.0 - u[..., 0]))
    phi = 2.0 * math.pi * u[..., 1]
    q0 = -torch.log(u[..., 2] * u[..., 3])
    q = torch.stack([q0, q0 * s * torch.cos(phi), q0 * s * torch.sin(phi), q0 * c], -1)
    Q = q.sum(1, keepdim=True)
    M = torch.sqrt(Q[..., 0] ** 2 - (Q[..., 1:] ** 2).sum(-1))[..., None]
    b, gam, x = -Q[..., 1:] / M, Q[..., :1] / M, sqrts / M
    bq = (b * q[..., 1:]).sum(-1, keepdim=True)
    p = torch.cat([x * (gam * q[..., :1] + bq), x * (q[..., 1:] + b * q[..., :1] + bq * b / (1.0 + gam))], -1)
    m2 = torch.zeros(nf, dtype=u.dtype, device=u.device)
    m2[:2] = mt * mt
    e0 = p[..., 0]
    xi = torch.full((u.shape[0], 1), math.sqrt(1.0 - (2.0 * mt / sqrts) ** 2), dtype=u.dtype, device=u.device)
    for _ in range(12):
        e = torch.sqrt(m2 + (xi * e0) ** 2)
        xi = xi - (e.sum(1, keepdim=True) - sqrts) / (xi * e0 * e0 / e).sum(1, keepdim=True)
    e = torch.sqrt(m2 + (xi * e0) ** 2)
    v = xi * e0
    out = torch.zeros(u.shape[0], nf + 2, 4, dtype=u.dtype, device=u.device)
    out[:, :2, 0] = 0.5 * sqrts
    out[:, 0, 3], out[:, 1, 3] = 0.5 * sqrts, -0.5 * sqrts
    out[:, 2:, 0] = e
    out[:, 2:, 1:] = xi[..., None] * p[..., 1:]
    w0 = ((2.0 * math.pi) ** (4 - 3 * nf) * (math.pi / 2.0) ** (nf - 1) * (sqrts * sqrts) ** (nf - 2)
          / (math.factorial(nf - 1) * math.factorial(nf - 2)))
    wgt = w0 * xi[:, 0] ** (2 * nf - 3) * (v / e).prod(1) * sqrts / (v * v / e).sum(1)
    return out, wgt


def _philox_uniforms(seed, nevt, nf, dev):
    """Philox4x32-10 (Salmon et al.), counter {e_lo, e_hi, j, 0}, key {seed_lo, seed_hi}; u = (x + 1/2) 2^-32."""
    m32 = 0xFFFFFFFF
    e = torch.arange(nevt, dtype=torch.int64, device=dev)[:, None].expand(nevt, nf)
    j = torch.arange(nf, dtype=torch.int64, device=dev)[None, :].expand(nevt, nf)
    c = [e & m32, e >> 32, j, torch.zeros_like(j)]
    k0, k1 = seed & m32, (seed >> 32) & m32

    def mul(a, x):   # 32 x 32 -> (high, low) words
        xl, xh = x & 0xFFFF, x >> 16
        lo, hi = a * xl, a * xh
        t = (lo >> 16) + hi
        return t >> 16, ((t & 0xFFFF) << 16) | (lo & 0xFFFF)

    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c[0])
        h1, l1 = mul(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & m32, (k1 + 0xBB67AE85) & m32
    return (torch.stack(c, -1).to(torch.float64) + 0.5) * 2.0 ** -32


def _inputs(case, seed, dev):
    """Momenta [nevt, npar, 4] and, for the epilogue, two uniforms per event."""
    g = torch.Generator(device=dev)
    g.manual_seed(1_000_003 * (seed + 1) + case["nevt"])
    nf = NG[case["process"]] + 2
    u = torch.rand(case["nevt"], nf, 4, generator=g, dtype=torch.float64, device=dev).clamp_(1e-12, 1.0 - 1e-12)
    r = torch.rand(2, case["nevt"], generator=g, dtype=torch.float64, device=dev)
    return _rambo(u)[0], r


def _pages(mom):
    """[nevt, npar, 4] -> the engine's AoSoA pages of 32 events (mg.h), zero padded."""
    n, npar, _ = mom.shape
    pages = (n + 31) // 32
    buf = torch.zeros(pages * 32, npar, 4, dtype=mom.dtype, device=mom.device)
    buf[:n] = mom
    return buf.reshape(pages, 32, npar, 4).permute(0, 2, 3, 1).contiguous().reshape(-1)


def _philox_seed(case, seed):
    return 7919 * (seed + 1) + case["nevt"]


def prepare(case, seed):
    n, kind = case["nevt"], case["kind"]
    ctx = mg.Context(case["process"])
    st = {"case": case, "ctx": ctx, "mode": MODES[case["mode"]]}
    f64 = dict(dtype=torch.float64, device="cuda")
    if kind == "step":
        st["seed"] = _philox_seed(case, seed)
        st["mom"] = torch.zeros(ctx.mom_count(n), **f64)
        st["wgt"], st["me"] = torch.zeros(n, **f64), torch.zeros(n, **f64)
        return st
    mom, r = _inputs(case, seed, torch.device("cuda"))
    st["mom"] = _pages(mom)
    st["me"] = torch.zeros(n, **f64)
    if kind == "host":
        st["mom"] = st["mom"].cpu().pin_memory()
        st["me"] = torch.zeros(n, dtype=torch.float64).pin_memory()
    elif kind == "lhe":
        st["rnd"] = r
        st["hel"] = torch.zeros(n, dtype=torch.int32, device="cuda")
        st["col"] = torch.zeros(n, dtype=torch.int32, device="cuda")
        st["as"] = torch.zeros(n, **f64)
    elif kind == "sde":
        st["w"] = torch.zeros(len(mg.sde_channels(case["process"])) * n, **f64)
    torch.cuda.synchronize()
    return st


def run(st):
    ctx, n, kind, mode = st["ctx"], st["case"]["nevt"], st["case"]["kind"], st["mode"]
    if kind == "me":
        ctx.sigmakin(st["mom"], n, st["me"], mode)
        return st["me"]
    if kind == "step":
        ctx.rambo(st["seed"], n, SQRTS, st["mom"], st["wgt"])
        ctx.hel_filter(st["mom"], min(n, 1024))
        ctx.sigmakin(st["mom"], n, st["me"], mode)
        return {"mom": st["mom"], "wgt": st["wgt"], "me": st["me"]}
    if kind == "host":
        ctx.sigmakin_host(st["mom"], n, st["me"], mode)
        return st["me"]
    if kind == "lhe":
        ctx.sigmakin_lhe(st["mom"], n, st["me"], st["rnd"][0], st["rnd"][1], st["hel"], st["col"],
                         running_alphas=True, alphas=st["as"])
        return {"me": st["me"], "hel": st["hel"], "col": st["col"], "alphas": st["as"]}
    ctx.sde_weights(st["mom"], n, st["w"])
    return st["w"]


def _nchannels(K):
    return {2: 3, 3: 15, 4: 105, 5: 945}[K]


def work(case):
    """Inputs and outputs once.  Operations: per colour ordering and helicity configuration one product
    with the antitop spinor per gluon on the quark line (32 flops a row spinor times a spinor), and the
    colour sum's multiply-adds on the orderings once; configurations with every helicity flipped have the
    same |M|^2 and count once."""
    n, K = case["nevt"], NG[case["process"]] + 2
    hel, ncol = 2 ** (K + 1), math.factorial(K)
    nbytes = 8 * (4 * (K + 2) + 1)
    flops = hel * ncol * (32.0 * K + 8.0)
    if case["kind"] == "step":
        nbytes += 8
    elif case["kind"] == "lhe":
        nbytes += 2 * 8 + 2 * 4 + 8
    elif case["kind"] == "sde":
        nbytes += 8 * (_nchannels(K) - 1)
        flops = hel * _nchannels(K) * (32.0 + 4.0)
    return {"bytes": float(n * nbytes), "flops": float(n * flops)}


# ------------------------------------------------------------------------------------------
# the same outputs in plain torch, 64 bits
# ------------------------------------------------------------------------------------------
def _dot(a, b):
    return a[..., 0, :] * b[..., 0, :] - a[..., 1, :] * b[..., 1, :] - a[..., 2, :] * b[..., 2, :] - a[..., 3, :] * b[..., 3, :]


def _slash_row(s, J):
    """Row spinor times gamma.J, chiral basis: s[..., 4, n], J[..., 4, n]."""
    a, b = J[..., 0, :] + J[..., 3, :], J[..., 0, :] - J[..., 3, :]
    jm, jp = J[..., 1, :] - 1j * J[..., 2, :], J[..., 1, :] + 1j * J[..., 2, :]
    s0, s1, s2, s3 = (s[..., i, :] for i in range(4))
    return torch.stack([s2 * a + s3 * jp, s2 * jm + s3 * b, s0 * b - s1 * jp, s1 * a - s0 * jm], -2)


class _Event:
    """Wavefunctions and propagators of a chunk of events: component index before the event index."""

    def __init__(self, mom):
        n, npar, _ = mom.shape
        self.n, self.K, self.dev = n, npar - 2, mom.device
        p = mom.permute(1, 2, 0)
        g = [0, 1] + list(range(4, npar))
        self.pin = [p[i] if i < 2 else -p[i] for i in g]          # momenta flowing in
        self.pt = p[2]
        self.gs = math.sqrt(4.0 * math.pi * ALPHAS)
        self.eps = [self._gluon(p[i], i >= 2) for i in g]
        self.ub, self.v = self._tops(p[2], p[3])
        self.P = {0: torch.zeros(4, n, dtype=mom.dtype, device=mom.device)}
        for S in range(1, 1 << self.K):
            low = (S & -S).bit_length() - 1
            self.P[S] = self.P[S & (S - 1)] + self.pin[low]

    def _gluon(self, k, outgoing):
        kt = torch.sqrt(k[1] ** 2 + k[2] ** 2)
        ka = torch.sqrt(kt ** 2 + k[3] ** 2)
        axis = kt == 0.0
        safe = torch.where(axis, torch.ones_like(kt), kt)
        cx = torch.where(axis, torch.where(k[3] < 0, -torch.ones_like(kt), torch.ones_like(kt)), k[1] * k[3] / (ka * safe))
        cy = torch.where(axis, torch.zeros_like(kt), k[2] * k[3] / (ka * safe))
        et = torch.stack([torch.zeros_like(kt), cx, cy, torch.where(axis, torch.zeros_like(kt), -kt / ka)])
        ep = torch.stack([torch.zeros_like(kt), torch.where(axis, torch.zeros_like(kt), -k[2] / safe),
                          torch.where(axis, torch.ones_like(kt), k[1] / safe), torch.zeros_like(kt)])
        sg = 1.0 if outgoing else -1.0
        return torch.stack([torch.complex(-lam * et, sg * ep) / math.sqrt(2.0) for lam in (-1.0, 1.0)])

    @staticmethod
    def _chi(p, lam):
        pa = torch.sqrt(p[1] ** 2 + p[2] ** 2 + p[3] ** 2)
        apz = torch.where(p[3] >= 0, pa + p[3], (p[1] ** 2 + p[2] ** 2) / (pa - p[3]).clamp_min(1e-300))
        nrm = torch.rsqrt(2.0 * pa * apz)
        up, low = torch.complex(apz * nrm, torch.zeros_like(pa)), torch.complex(p[1] * nrm, p[2] * nrm)
        return (up, low) if lam > 0 else (-low.conj(), up)

    def _tops(self, t, tb):
        ub, v = [], []
        for lam in (-1, 1):
            pa = torch.sqrt(t[1] ** 2 + t[2] ** 2 + t[3] ** 2)
            sp = torch.sqrt(t[0] + pa)
            sm = MT / sp
            c = self._chi(t, lam)
            fl, fr = (sm, sp) if lam > 0 else (sp, sm)
            ub.append(torch.stack([fr * c[0].conj(), fr * c[1].conj(), fl * c[0].conj(), fl * c[1].conj()]))
            pa = torch.sqrt(tb[1] ** 2 + tb[2] ** 2 + tb[3] ** 2)
            sp = torch.sqrt(tb[0] + pa)
            sm = MT / sp
            c = self._chi(tb, -lam)
            fl, fr = (-sp, sm) if lam > 0 else (sm, -sp)
            v.append(torch.stack([fl * c[0], fl * c[1], fr * c[0], fr * c[1]]))
        return torch.stack(ub), torch.stack(v)

    def gprop(self, S):
        P = self.P[S]
        return -self.gs / (P[0] ** 2 - P[1] ** 2 - P[2] ** 2 - P[3] ** 2)

    def quark(self, s, S):
        """s (Qslash + m) (-g) / (Q^2 - m^2), Q = p_t - P_S."""
        Q = self.pt - self.P[S]
        f = -self.gs / (Q[0] ** 2 - Q[1] ** 2 - Q[2] ** 2 - Q[3] ** 2 - MT * MT)
        return (_slash_row(s, Q.to(s.dtype)) + MT * s) * f


def _v3(JL, JR, PL, PR, full):
    """Three-gluon vertex; full: also the terms that vanish between conserved currents."""
    d = PL - PR
    a, b = (PL + 2.0 * PR, 2.0 * PL + PR) if full else (2.0 * PR, 2.0 * PL)
    ct = JL.dtype
    return (d.to(ct) * _dot(JL, JR)[..., None, :] + _dot(JL, a.to(ct))[..., None, :] * JR
            - _dot(JR, b.to(ct))[..., None, :] * JL)


def _v4(A, B, C):
    return (_dot(A, B)[..., None, :] * C + _dot(B, C)[..., None, :] * A - 2.0 * _dot(A, C)[..., None, :] * B)


def _jamps(mom):
    """Colour-ordered amplitudes {ordering: [2^K gluon helicities (ordering's axes), t, tbar, n]}."""
    ev = _Event(mom)
    K, n = ev.K, ev.n
    mask = lambda seq: sum(1 << g for g in seq)
    J = {(g,): ev.eps[g] for g in range(K)}

    def ax(x, before, after):   # helicity axes of a sub-sequence inside a longer one
        return x.reshape((1,) * before + x.shape[:-2] + (1,) * after + x.shape[-2:])

    for L in range(2, K + 1):
        for seq in itertools.permutations(range(K), L):
            if seq > seq[::-1]:
                r = J[seq[::-1]]
                J[seq] = (-1.0) ** (L + 1) * r.permute(*range(L - 1, -1, -1), L, L + 1)
                continue
            acc = 0
            for i in range(1, L):
                acc = acc + _v3(ax(J[seq[:i]], 0, L - i), ax(J[seq[i:]], i, 0), ev.P[mask(seq[:i])], ev.P[mask(seq[i:])], False)
                for k in range(i + 1, L):
                    acc = acc + ev.gs * _v4(ax(J[seq[:i]], 0, L - i), ax(J[seq[i:k]], i, L - k), ax(J[seq[k:]], k, 0))
            J[seq] = acc * ev.gprop(mask(seq))
    psi = {(): ev.ub}          # [t, helicities..., 4, n]
    out = {}
    for L in range(1, K + 1):
        for seq in itertools.permutations(range(K), L):
            acc = 0
            for i in range(L):
                s = psi[seq[:i]]
                s = s.reshape(s.shape[:-2] + (1,) * (L - i) + s.shape[-2:])
                acc = acc + _slash_row(s, ax(J[seq[i:]], i, 0)[None])
            if L < K:
                psi[seq] = ev.quark(acc, mask(seq))
            else:
                a = torch.stack([(acc * ev.v[b]).sum(-2) for b in range(2)], -2)   # [t, hel..., tbar, n]
                # helicity axes from the ordering's positions to gluon labels
                inv = [seq.index(g) for g in range(K)]
                out[seq] = a.permute(*[1 + q for q in inv], 0, K + 1, K + 2)
    return out


def _colour(K):
    """Tr(T^s1 .. T^sK T^tK .. T^t1) over all colours, orderings in lexicographic order."""
    lam = np.zeros((8, 3, 3), complex)
    lam[0][0, 1] = lam[0][1, 0] = 1
    lam[1][0, 1], lam[1][1, 0] = -1j, 1j
    lam[2][0, 0], lam[2][1, 1] = 1, -1
    lam[3][0, 2] = lam[3][2, 0] = 1
    lam[4][0, 2], lam[4][2, 0] = -1j, 1j
    lam[5][1, 2] = lam[5][2, 1] = 1
    lam[6][1, 2], lam[6][2, 1] = -1j, 1j
    lam[7] = np.diag([1, 1, -2]) / math.sqrt(3.0)
    T = lam / 2.0
    prod = np.eye(3, dtype=complex)
    for i in range(K):
        prod = np.einsum("...ij,ajk->...aik", prod, T)
    perms = list(itertools.permutations(range(K)))
    rank = {s: i for i, s in enumerate(perms)}
    # the product along ordering s has colour index a_s[i] on matrix i: axis g of the tensor in gluon labels
    # is position s.index(g); only the relative ordering matters
    rel = np.empty(len(perms))
    for s in perms:
        axes = tuple(s.index(g) for g in range(K))
        rel[rank[s]] = np.sum(prod * np.conj(prod.transpose(axes + (K, K + 1)))).real
    C = np.empty((len(perms), len(perms)))
    for i, s in enumerate(perms):
        where = {g: q for q, g in enumerate(s)}
        for j, t in enumerate(perms):
            C[i, j] = rel[rank[tuple(where[g] for g in t)]]
    return C


def _helicity_sums(mom):
    """|M_h|^2 summed over colours [nhel, n] (helicity index: bits g1 g2 t tbar g3 .., g1 highest) and the
    flow weights sum_h |A_flow|^2 [ncol, n]."""
    A = _jamps(mom)
    K, n = mom.shape[1] - 2, mom.shape[0]
    seqs = sorted(A)
    # axes (gluons 0 .. K-1, t, tbar, n) -> particle order
    order = [0, 1, K, K + 1] + list(range(2, K)) + [K + 2]
    jam = torch.stack([A[s].permute(*order).reshape(-1, n) for s in seqs])     # [ncol, nhel, n]
    del A
    C = torch.tensor(_colour(K), dtype=torch.float64, device=mom.device)
    ncol = len(seqs)
    gs2 = 4.0 * math.pi * ALPHAS
    tot = 0.0
    for part in (jam.real.contiguous().reshape(ncol, -1), jam.imag.contiguous().reshape(ncol, -1)):
        tot = tot + (part * (C @ part)).sum(0)
    flow = (jam.real ** 2 + jam.imag ** 2).sum(1)
    return gs2 * tot.reshape(-1, n), flow


def _chunks(mom):
    K = mom.shape[1] - 2
    step = {2: 131072, 3: 65536, 4: 32768, 5: 8192}[K]
    return [mom[i:i + step] for i in range(0, mom.shape[0], step)]


def _channel_weights(mom):
    """Channel weights [nch, n]: sum_h |A_d|^2 normalised over the channels, channels in the engine's order
    (the first tree's gluon subset descending, trees of a subset as below, depth first)."""
    ev = _Event(mom)
    K, n = ev.K, ev.n
    trees = {1 << g: [((g,), ev.eps[g])] for g in range(K)}
    by_size = sorted((S for S in range(1, 1 << K) if S & (S - 1)), key=lambda S: (bin(S).count("1"), S))
    for S in by_size:
        trees[S] = []
        A = (S - 1) & S
        while A:
            if A & (S & -S):
                B = S ^ A
                for ga, ja in trees[A]:
                    for gb, jb in trees[B]:
                        JL = ja.reshape(ja.shape[:-2] + (1,) * len(gb) + ja.shape[-2:])
                        JR = jb.reshape((1,) * len(ga) + jb.shape)
                        trees[S].append((ga + gb, _v3(JL, JR, ev.P[A], ev.P[B], True) * ev.gprop(S)))
            A = (A - 1) & S
    out = []

    def walk(rem, psi, used, done):
        S = rem
        while S:
            for gl, J in trees[S]:
                s = psi.reshape(psi.shape[:-2] + (1,) * len(gl) + psi.shape[-2:])
                r = _slash_row(s, J.reshape((1,) * (1 + used) + J.shape))
                if S == rem:
                    out.append(sum((((r * ev.v[b]).sum(-2).abs()) ** 2).reshape(-1, n).sum(0) for b in range(2)))
                else:
                    walk(rem ^ S, ev.quark(r, done | S), used + len(gl), done | S)
            S = (S - 1) & rem

    walk((1 << K) - 1, ev.ub, 0, 0)
    w = torch.stack(out)
    return w / w.sum(0)


def exact(case, seed):
    dev = _device()
    ng, n, kind = NG[case["process"]], case["nevt"], case["kind"]
    if kind == "step":
        mom, wgt = _rambo(_philox_uniforms(_philox_seed(case, seed), n, ng + 2, dev))
    else:
        mom, r = _inputs(case, seed, dev)
    if kind == "sde":
        return torch.cat([_channel_weights(m) for m in _chunks(mom)], 1).reshape(-1)
    norm = 1.0 / (256.0 * math.factorial(ng))
    me, hel, col, als, at = [], [], [], [], 0
    for m in _chunks(mom):
        mh, flow = _helicity_sums(m)
        total = mh.sum(0) * norm
        if kind == "lhe":
            k = slice(at, at + m.shape[0])
            at += m.shape[0]

            def pick(w, u):
                cum = torch.cumsum(w, 0)
                return (cum <= u * cum[-1]).sum(0).clamp_max(w.shape[0] - 1).to(torch.int32)

            hel.append(pick(mh, r[0, k]))
            col.append(pick(flow, r[1, k]))
            mt2 = torch.zeros(m.shape[1] - 2, dtype=m.dtype, device=m.device)
            mt2[:2] = MT * MT
            mu = 0.5 * torch.sqrt(mt2 + m[:, 2:, 1] ** 2 + m[:, 2:, 2] ** 2).sum(1)
            b0 = (33.0 - 2.0 * 5) / (12.0 * math.pi)
            a = ALPHAS / (1.0 + ALPHAS * b0 * torch.log(mu * mu / 91.1876 ** 2))
            als.append(a)
            total = total * (a / ALPHAS) ** (ng + 2)
        me.append(total)
    me = torch.cat(me)
    if kind == "lhe":
        return {"me": me, "hel": torch.cat(hel), "col": torch.cat(col), "alphas": torch.cat(als)}
    if kind == "step":
        return {"mom": _pages(mom), "wgt": wgt, "me": me}
    return me.cpu() if kind == "host" else me
