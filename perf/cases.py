"""What a user of the library has it do, as cases that can be timed and checked.

A case is a dict of plain values.  Its "kind" is one way of using the library:

* ``apply``          out = Mhat^dag Mhat in on native device buffers: the operator call inside a caller's own
                     Krylov loop, at each storage precision and option (12- or 18-real links, FP64 units or
                     double-float, chemical potential, U(1) phases);
* ``apply_batch``    the same for many right-hand sides of one lattice (a block solver's operator) or for a
                     ragged set of lattices, in one call;
* ``canonical``      Mhat (or Mhat^dag) of a spinor in the caller's own layout: convert, apply, convert back, the
                     way an analysis code calls the operator once;
* ``configuration``  what a new gauge configuration costs before its first solve: set the links, build the clover
                     term and its inverse, its log det, smear the links of the hopping term, first Mhat;
* ``solve``          one conjugate-gradient solve of Mhat^dag Mhat x = b, plain FP64 or mixed precision;
* ``multishift``     the shifted systems of a rational approximation in one solve.

Solves run to 1e-12, the residual of the energy evaluations in a trajectory's accept step.  Links are
exp(i eps A), A Gaussian traceless Hermitian, projected onto SU(3); sources are Gaussian.
"""
import math

import numpy as np
import torch

from paper_1711_03836_gb300 import bqcd

# ---------------------------------------------------------------------------- the cases

_SHIFTS = [10.0 ** (-4.0 + 4.0 * k / 9.0) for k in range(10)]


def _case(kind, dims, **more):
    c = {"kind": kind, "lx": dims[0], "ly": dims[1], "lz": dims[2], "lt": dims[3], "eps": 0.2, "kappa": 0.135,
         "csw": 1.7, "mu": 0.0, "prec": "single", "recon": 12, "arith": "df64"}
    c.update(more)
    return c


def listed():
    return [
        # the smallest lattice: a handful of thread blocks per launch, launches and latency are everything
        _case("apply", (8, 8, 8, 8), name="apply_single_8x8x8x8", eps=0.3, kappa=0.125, csw=1.0),
        # the plain FP64 solver in the library's default arithmetic, on the small lattice it is tested on
        _case("solve", (8, 8, 8, 8), name="cg_double_8x8x8x8", eps=0.3, kappa=0.125, csw=1.0, prec="double",
              recon=18, arith="native", iterations=72),
        # four lattices of uneven volume in one call (ensembles of several volumes, finite-size studies)
        _case("apply_batch", (20, 20, 20, 40), name="apply_batch_ragged", ragged=True, nrhs=4),
        # FP64 on the FP64 units with a chemical potential, the reference arithmetic of a small production run
        _case("apply", (16, 16, 16, 32), name="apply_double_16x16x16x32", mu=0.1, prec="double", recon=18,
              arith="native"),
        # the rational approximation's ten shifted systems
        _case("multishift", (16, 16, 16, 32), name="multishift_16x16x16x32", iterations=130),
        # one operator application on a spinor in the caller's layout, on a lattice of unequal, odd-factor extents
        _case("canonical", (18, 14, 22, 30), name="canonical_double_18x14x22x30", mu=0.1, prec="double", recon=12,
              dagger=True),
        # double-float FP64: the reliable updates and FP64 Krylov spaces of production solves
        _case("apply", (24, 24, 24, 48), name="apply_df64_24x24x24x48", prec="double", recon=18),
        # twelve spin-colour sources of a propagator, block solver's operator
        _case("apply_batch", (24, 24, 24, 48), name="apply_batch12_24x24x24x48", ragged=False, nrhs=12),
        # a new configuration of a trajectory, with stout-smeared hopping links
        _case("configuration", (24, 24, 24, 48), name="configuration_24x24x24x48", rho=0.1),
        # FP16 storage with per-site scales on a production volume
        _case("apply", (32, 32, 32, 64), name="apply_half_32x32x32x64", eps=0.15, kappa=0.1355, csw=1.9, prec="half"),
        # the production solve: FP32 inner iteration, double-float reliable updates
        _case("solve", (32, 32, 32, 64), name="cg_mixed_32x32x32x64", eps=0.15, kappa=0.1355, csw=1.9,
              iterations=112),
        # the largest lattice, with the U(1) phases of a charged flavour (18-real links)
        _case("apply", (48, 48, 48, 96), name="apply_single_qed_48x48x48x96", eps=0.15, kappa=0.1355, csw=1.9,
              recon=18, charge=2.0 / 3.0),
    ]


def _draw_dims(rng, lo, hi):
    """Four even extents >= 4, often unequal and with odd factors, whose product lies in [lo, hi]."""
    while True:
        target = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        side = target ** 0.25
        d = [max(4, 2 * round(side * math.exp(rng.uniform(-0.35, 0.35)) / 2)) for _ in range(3)]
        t = max(4, 2 * round(target / (d[0] * d[1] * d[2]) / 2))
        if t <= 128 and lo <= d[0] * d[1] * d[2] * t <= hi:
            return (d[0], d[1], d[2], t)


def draw(rng):
    kind = rng.choice(["apply", "apply", "apply", "apply_batch", "canonical", "configuration", "solve", "multishift"])
    mu = rng.choice([0.0, 0.0, 0.1])
    eps = rng.choice([0.15, 0.2, 0.3])
    coupling = {"eps": eps, "mu": mu}
    coupling.update({0.15: {"kappa": 0.1355, "csw": 1.9}, 0.2: {"kappa": 0.135, "csw": 1.7},
                     0.3: {"kappa": 0.125, "csw": 1.0}}[eps])
    if kind == "apply":
        prec = rng.choice(["double", "single", "single", "half"])
        arith = rng.choice(["native", "df64"])
        charge = rng.choice([0.0, 0.0, 2.0 / 3.0, -1.0 / 3.0])
        recon = 18 if charge else rng.choice([12, 18])
        more = {"prec": prec, "arith": arith, "recon": recon}
        if charge:
            more["charge"] = charge
        return _case(kind, _draw_dims(rng, 4096, 2 ** 21 if prec == "double" else 2 ** 23), **coupling, **more)
    if kind == "apply_batch":
        return _case(kind, _draw_dims(rng, 4096, 700_000), ragged=False, nrhs=rng.randrange(2, 17),
                     prec=rng.choice(["single", "single", "half"]), **coupling)
    if kind == "canonical":
        return _case(kind, _draw_dims(rng, 4096, 2 ** 20), prec="double", recon=rng.choice([12, 18]),
                     arith=rng.choice(["native", "df64"]), dagger=rng.choice([False, True]), **coupling)
    if kind == "configuration":
        return _case(kind, _draw_dims(rng, 4096, 700_000), rho=rng.choice([0.05, 0.1]), **coupling)
    if kind == "solve":
        prec = rng.choice(["double", "single", "single"])
        return _case(kind, _draw_dims(rng, 4096, 400_000), prec=prec, recon=18 if prec == "double" else 12,
                     iterations=100, **coupling)
    return _case(kind, _draw_dims(rng, 4096, 140_000), iterations=130, **coupling)


# ---------------------------------------------------------------------------- inputs

_RAGGED = [(8, 8, 8, 8), (12, 12, 12, 12), (16, 16, 16, 32), (20, 20, 20, 40)]


def _dims(case):
    return (case["lx"], case["ly"], case["lz"], case["lt"])


def _volume(dims):
    return dims[0] * dims[1] * dims[2] * dims[3]


def _lattices(case):
    return _RAGGED if case.get("ragged") else [_dims(case)]


def _generator(seed, what):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1009 + what) % (2 ** 63))
    return g


def _links(dims, eps, seed, what=0):
    """[V][4][3][3] complex128: exp(i eps A) to third order, rows orthonormalised, third row from the first two."""
    n = _volume(dims) * 4
    g = _generator(seed, what)
    out = torch.empty((n, 3, 3), dtype=torch.complex128, device="cuda")
    step = 1 << 22
    for a in range(0, n, step):
        m = min(step, n - a)
        w = torch.randn((8, m), generator=g, device="cuda", dtype=torch.float32).double() * (0.5 * eps)
        w8 = w[7] / math.sqrt(3.0)
        H = [[torch.complex(w8 + w[2], torch.zeros_like(w8)), torch.complex(w[0], -w[1]), torch.complex(w[3], -w[4])],
             [torch.complex(w[0], w[1]), torch.complex(w8 - w[2], torch.zeros_like(w8)), torch.complex(w[5], -w[6])],
             [torch.complex(w[3], w[4]), torch.complex(w[5], w[6]), torch.complex(-2.0 * w8, torch.zeros_like(w8))]]

        def row(i):  # row i of 1 + iH - H^2/2 - i H^3/6
            h2 = [sum(H[i][k] * H[k][j] for k in range(3)) for j in range(3)]
            h3 = [sum(h2[k] * H[k][j] for k in range(3)) for j in range(3)]
            return [(1.0 if i == j else 0.0) + 1j * H[i][j] - 0.5 * h2[j] - (1j / 6.0) * h3[j] for j in range(3)]

        def unit(r):
            s = torch.rsqrt(sum(v.real ** 2 + v.imag ** 2 for v in r))
            return [v * s for v in r]

        r0, r1 = unit(row(0)), row(1)
        for _ in range(2):  # twice: orthogonal to the last bit
            p = sum(r0[k].conj() * r1[k] for k in range(3))
            r1 = unit([r1[k] - p * r0[k] for k in range(3)])
        o = out[a:a + m]
        for k in range(3):
            o[:, 0, k], o[:, 1, k] = r0[k], r1[k]
            i, j = (k + 1) % 3, (k + 2) % 3
            o[:, 2, k] = (r0[i] * r1[j] - r0[j] * r1[i]).conj()
    return out.reshape(-1, 4, 3, 3)


def _angles(dims, seed):
    return 0.1 * torch.randn((_volume(dims), 4), generator=_generator(seed, 7), device="cuda", dtype=torch.float64)


def _spinor(dims, seed, what, single):
    """[V/2][4][3] complex128, Gaussian; `single`: values that FP32 holds."""
    z = torch.randn((_volume(dims) // 2, 4, 3, 2), generator=_generator(seed, 100 + what), device="cuda",
                    dtype=torch.float32 if single else torch.float64).double()
    return torch.view_as_complex(z)


def _lattice(case, dims, seed, what=0):
    lat = bqcd.Lattice(dims, case["kappa"], case["csw"], case["mu"], -1.0, case.get("charge", 0.0))
    bqcd.bq_set_fp64_arith(lat.ctx, case["arith"])
    bqcd.bq_set_recon(lat.ctx, case["prec"], case["recon"])
    bqcd.bq_set_gauge(lat.ctx, _links(dims, case["eps"], seed, what))
    if case.get("charge"):
        bqcd.bq_set_u1(lat.ctx, _angles(dims, seed))
    return lat


def _values(buf, prec, vh):
    """A native spinor buffer as the numbers it holds."""
    if prec == "double":
        return buf.view(torch.float64)
    if prec == "single":
        return buf.view(torch.float32)
    return [buf[:48 * vh].view(torch.float16), buf[48 * vh:].view(torch.float32)]


def prepare(case, seed):
    kind, dims, prec = case["kind"], _dims(case), case["prec"]
    s = {"case": case}
    if kind == "apply_batch":
        lats = [_lattice(case, d, seed, 10 * k) for k, d in enumerate(_lattices(case))]
        ctxs = lats if case["ragged"] else lats * case["nrhs"]
        s["lats"], s["ctxs"] = ctxs, [x.ctx for x in ctxs]
        s["ins"] = [x.pack(_spinor(x.dims, seed, k, True), prec) for k, x in enumerate(ctxs)]
        s["outs"] = [x.spinor(prec) for x in ctxs]
        for x in lats:
            bqcd.bq_build_clover(x.ctx)
        return s
    if kind == "configuration":
        lat = bqcd.Lattice(dims, case["kappa"], case["csw"], case["mu"], -1.0)
        bqcd.bq_set_recon(lat.ctx, "single", 12)
        bqcd.bq_set_stout(lat.ctx, case["rho"], 1)
        s["lat"], s["links"] = lat, _links(dims, case["eps"], seed)
        s["hop"] = torch.empty_like(s["links"])
        s["in"], s["out"] = lat.pack(_spinor(dims, seed, 0, True), "single"), lat.spinor("single")
        return s
    s["lat"] = lat = _lattice(case, dims, seed)
    bqcd.bq_build_clover(lat.ctx)
    psi = _spinor(dims, seed, 0, prec != "double")
    if kind == "apply":
        s["in"], s["out"] = lat.pack(psi, prec), lat.spinor(prec)
    elif kind == "canonical":
        s["psi"], s["res"], s["in"], s["out"] = psi, torch.empty_like(psi), lat.spinor(prec), lat.spinor(prec)
    else:
        s["b"] = psi
        s["x"] = [torch.empty_like(psi) for _ in range(10 if kind == "multishift" else 1)]
    return s


def run(s):
    case = s["case"]
    kind, prec = case["kind"], case["prec"]
    if kind == "apply":
        bqcd.bq_apply_mdagm(s["lat"].ctx, s["out"], s["in"], prec)
        return _values(s["out"], prec, s["lat"].Vh)
    if kind == "apply_batch":
        bqcd.bq_apply_mdagm_batch(s["ctxs"], s["outs"], s["ins"], prec)
        return [_values(o, prec, x.Vh) for o, x in zip(s["outs"], s["lats"])]
    ctx = s["lat"].ctx
    if kind == "canonical":
        bqcd.bq_spinor_pack(ctx, s["in"], s["psi"], prec)
        bqcd.bq_apply_mhat(ctx, s["out"], s["in"], case["dagger"], prec)
        bqcd.bq_spinor_unpack(ctx, s["res"], s["out"], prec)
        return s["res"]
    if kind == "configuration":
        bqcd.bq_set_gauge(ctx, s["links"])
        bqcd.bq_build_clover(ctx)
        logdet, _ = bqcd.bq_clover_logdet(ctx, 1)
        bqcd.bq_get_hop_links(ctx, s["hop"])
        bqcd.bq_apply_mhat(ctx, s["out"], s["in"], 0, "single")
        return {"logdet": np.array([logdet]), "links": s["hop"], "mhat": _values(s["out"], "single", s["lat"].Vh)}
    if kind == "solve":
        bqcd.bq_solve_cg(ctx, s["x"][0], s["b"], tol=1e-12, precision=prec, delta=1e-3)
        return s["x"][0]
    bqcd.bq_solve_multishift_cg(ctx, s["x"], s["b"], _SHIFTS, tol=1e-12, precision=prec, delta=1e-3)
    return s["x"]


# ---------------------------------------------------------------------------- what a pass cannot do without

def work(case):
    """Each field and vector once: links of both parities, A on the even and A^-1 on the odd sites, the vectors."""
    kind = case["kind"]
    size = {"double": 8.0, "single": 4.0, "half": 2.0}[case["prec"]]
    spinor = 24.0 * size + (4.0 if case["prec"] == "half" else 0.0)
    fields = 8.0 * case["recon"] * size + 144.0 * size  # per site of one parity
    mdagm = 2.0 * (1320.0 + 504.0) + 2.0 * (1320.0 + 504.0 + 48.0)
    if kind == "apply_batch" and case["ragged"]:
        vh = sum(_volume(d) // 2 for d in _RAGGED)
        return {"bytes": vh * (fields + 2.0 * spinor), "flops": vh * mdagm}
    vh = _volume(_dims(case)) // 2
    if kind == "apply":
        return {"bytes": vh * (fields + 2.0 * spinor), "flops": vh * mdagm}
    if kind == "apply_batch":
        return {"bytes": vh * (fields + 2.0 * spinor * case["nrhs"]), "flops": vh * mdagm * case["nrhs"]}
    if kind == "canonical":
        return {"bytes": vh * (fields + 2.0 * 192.0), "flops": vh * 0.5 * mdagm}
    if kind == "configuration":
        # links read and smeared links written (FP64), vectors in FP32; per site six planes of four leaves (three
        # 3x3 products each), four links of six staples (two products each), two 6x6 inverses
        prod = 27.0 * 8.0
        return {"bytes": 2.0 * vh * 2.0 * 576.0 + vh * 192.0,
                "flops": 2.0 * vh * (72.0 * prod + 48.0 * prod + 8.0 * prod + 2.0 * 6.0 ** 3 * 8.0)}
    solutions = 10.0 if kind == "multishift" else 1.0
    return {"bytes": vh * (fields + 192.0 * (1.0 + solutions)),
            "flops": vh * case["iterations"] * (mdagm + 200.0 * solutions)}


# ---------------------------------------------------------------------------- the same in plain torch, 64 bits

# gamma_mu in the chiral basis: (gamma psi)_s = phase[s] psi_perm[s]
_PERM = [[3, 2, 1, 0], [3, 2, 1, 0], [2, 3, 0, 1], [2, 3, 0, 1]]
_PHASE = [[-1j, -1j, 1j, 1j], [-1, 1, 1, -1], [-1j, 1j, 1j, -1j], [1, 1, 1, 1]]


class _Exact:
    def __init__(self, case, dims, seed, what=0, links=None, hop=None):
        self.case, self.dims, self.V = case, dims, _volume(dims)
        self.vh = self.V // 2
        lex = torch.arange(self.V, device="cuda")
        self.x, r = [], lex
        for L in dims:
            self.x.append(r % L)
            r = r // L
        parity = sum(self.x) % 2
        self.sites = [lex[parity == p] for p in (0, 1)]
        U = _links(dims, case["eps"], seed, what) if links is None else links
        self.thin = U
        H = U if hop is None else hop
        if case.get("charge"):
            H = H * torch.exp(-1j * case["charge"] * _angles(dims, seed))[:, :, None, None]
        self.H = [[H[self.sites[p], mu].permute(1, 2, 0).contiguous() for mu in range(4)] for p in (0, 1)]
        A = self._clover()
        self.A = A[0]
        self.Ainv = self._inverse(A[1])
        del A

    def shift(self, mu, by):
        """lex index of the neighbour of every site"""
        L, stride = self.dims[mu], 1
        for k in range(mu):
            stride *= self.dims[k]
        lex = torch.arange(self.V, device="cuda")
        return lex + ((self.x[mu] + by) % L - self.x[mu]) * stride

    @staticmethod
    def mm(a, b):
        return torch.stack([torch.stack([a[i, 0] * b[0, j] + a[i, 1] * b[1, j] + a[i, 2] * b[2, j] for j in range(3)])
                            for i in range(3)])

    @staticmethod
    def dag(a):
        return a.transpose(0, 1).conj()

    def _clover(self):
        """[2][block][6][6][V/2] of the even and the odd sites."""
        kc = self.case["kappa"] * self.case["csw"]
        gam = []
        for mu in range(4):
            g = torch.zeros((4, 4), dtype=torch.complex128)
            for s in range(4):
                g[s, _PERM[mu][s]] = _PHASE[mu][s]
            gam.append(g)
        A = [torch.zeros((2, 6, 6, self.vh), dtype=torch.complex128, device="cuda") for _ in (0, 1)]
        for a in A:
            for i in range(6):
                a[:, i, i] = 1.0
        U = [self.thin[:, mu].permute(1, 2, 0).contiguous() for mu in range(4)]
        at = lambda m, idx: m[:, :, idx]  # noqa: E731
        for mu in range(4):
            for nu in range(mu + 1, 4):
                m, n = U[mu], U[nu]
                fm, fn = self.shift(mu, 1), self.shift(nu, 1)
                bm, bn = self.shift(mu, -1), self.shift(nu, -1)
                plaq = self.mm(self.mm(m, at(n, fm)), self.dag(self.mm(n, at(m, fn))))  # at x, plane mu nu
                Q = plaq
                # the other leaves are the neighbouring plaquettes, carried to x along their links
                mb, nb = at(m, bm), at(n, bn)
                Q = Q + self.mm(self.mm(self.dag(mb), at(plaq, bm)), mb)
                Q = Q + self.mm(self.mm(self.dag(nb), at(plaq, bn)), nb)
                bmn = bm[bn]
                path = self.mm(at(n, bmn), mb)
                Q = Q + self.mm(self.mm(self.dag(path), at(plaq, bmn)), path)
                F = (Q - self.dag(Q)) / 8.0
                tr = (F[0, 0] + F[1, 1] + F[2, 2]) / 3.0
                for k in range(3):
                    F[k, k] = F[k, k] - tr
                sigma = 0.5j * (gam[mu] @ gam[nu] - gam[nu] @ gam[mu])
                for p in (0, 1):
                    Fp = F[:, :, self.sites[p]]
                    for b in range(2):
                        for s in range(2):
                            for t in range(2):
                                v = complex(sigma[2 * b + s, 2 * b + t])
                                if v:
                                    A[p][b, 3 * s:3 * s + 3, 3 * t:3 * t + 3] += (1j * kc * v) * Fp
        return A

    def _inverse(self, A):
        """Gauss-Jordan in place on every block; the pivots' moduli give the log det."""
        A = A.clone()
        self.logdet = 0.0
        for k in range(6):
            p = 1.0 / A[:, k, k]
            self.logdet -= float(torch.log(p.abs()).sum())
            A[:, k, k] = 1.0
            row = A[:, k] * p[:, None]
            A[:, k] = row
            for i in range(6):
                if i != k:
                    f = A[:, i, k].clone()
                    A[:, i, k] = 0.0
                    A[:, i] -= f[:, None] * row
        return A

    @staticmethod
    def block(A, psi):
        v = psi.reshape(2, 6, -1)
        return torch.stack([sum(A[:, i, j] * v[:, j] for j in range(6)) for i in range(6)], 1).reshape(psi.shape)

    def hops(self, psi, p, dagger):
        """D_hop (or its adjoint) onto parity p; psi [4][3][V/2] lives on the other parity."""
        out = torch.zeros_like(psi)
        here = self.sites[p]
        mu_c = -self.case["mu"] if dagger else self.case["mu"]
        for mu in range(4):
            for by in (1, -1):
                n = self.shift(mu, by)[here] // 2
                sign = -by if not dagger else by  # (1 - gamma) forward in D, (1 + gamma) forward in the adjoint
                v = psi[:, :, n]
                h = torch.stack([v[s] + sign * _PHASE[mu][s] * v[_PERM[mu][s]] for s in range(4)])
                U = self.H[p][mu] if by > 0 else self.dag(self.H[1 - p][mu][:, :, n])
                w = torch.stack([U[i, 0] * h[:, 0] + U[i, 1] * h[:, 1] + U[i, 2] * h[:, 2] for i in range(3)], 1)
                if mu == 3:
                    edge = self.x[3][here] == (self.dims[3] - 1 if by > 0 else 0)
                    w = w * (math.exp(by * mu_c) * torch.where(edge, -1.0, 1.0).double())
                out += w
        return out

    def mhat(self, psi, dagger):
        odd = self.block(self.Ainv, self.hops(psi, 1, dagger))
        return self.block(self.A, psi) - self.case["kappa"] ** 2 * self.hops(odd, 0, dagger)

    def mdagm(self, psi):
        return self.mhat(self.mhat(psi, False), True)

    def solve(self, b, sigma=0.0):
        x, r = torch.zeros_like(b), b.clone()
        p, rr = r.clone(), float((r.abs() ** 2).sum())
        stop = 1e-28 * rr
        for _ in range(400):
            if rr <= stop:
                break
            q = self.mdagm(p) + sigma * p
            alpha = rr / float((p.conj() * q).real.sum())
            x += alpha * p
            r -= alpha * q
            new = float((r.abs() ** 2).sum())
            p = r + (new / rr) * p
            rr = new
        return x


def _in(psi):
    return psi.permute(1, 2, 0).contiguous()


def _native(v, prec):
    """[4][3][V/2] in the layout of the native buffers."""
    v = v.reshape(12, -1)
    if prec == "double":
        return torch.view_as_real(v.contiguous()).reshape(-1)
    if prec == "single":
        return torch.view_as_real(v.reshape(6, 2, -1).transpose(1, 2).contiguous()).reshape(-1)
    m = torch.maximum(v.real.abs(), v.imag.abs()).amax(0)
    return [torch.view_as_real((v / m).reshape(3, 4, -1).transpose(1, 2).contiguous()).reshape(-1), m]


def _smeared(U, dims, rho, shift):
    """One stout step of every link [V][4][3][3]."""
    L = [U[:, mu].permute(1, 2, 0).contiguous() for mu in range(4)]
    mm, dag = _Exact.mm, _Exact.dag
    out = torch.empty_like(U)
    for mu in range(4):
        C = 0
        fm = shift(mu, 1)
        for nu in range(4):
            if nu == mu:
                continue
            fn, bn = shift(nu, 1), shift(nu, -1)
            C = C + mm(mm(L[nu], L[mu][:, :, fn]), dag(L[nu][:, :, fm]))
            C = C + mm(mm(dag(L[nu][:, :, bn]), L[mu][:, :, bn]), L[nu][:, :, bn[fm]])
        W = rho * mm(C, dag(L[mu]))
        X = 0.5 * (W - dag(W))
        tr = (X[0, 0] + X[1, 1] + X[2, 2]) / 3.0
        E = torch.zeros_like(X)
        for k in range(3):
            X[k, k] = X[k, k] - tr
            E[k, k] = 1.0
        one = E.clone()
        for j in range(24, 0, -1):
            E = one + mm(X, E) / j
        out[:, mu] = mm(E, L[mu]).permute(2, 0, 1)
    return out


def exact(case, seed):
    kind, dims, prec = case["kind"], _dims(case), case["prec"]
    if kind == "apply_batch":
        lats = [_Exact(case, d, seed, 10 * k) for k, d in enumerate(_lattices(case))]
        lats = lats if case["ragged"] else lats * case["nrhs"]
        return [_native(x.mdagm(_in(_spinor(x.dims, seed, k, True))), prec) for k, x in enumerate(lats)]
    if kind == "configuration":
        U = _links(dims, case["eps"], seed)
        e = _Exact(case, dims, seed, links=U)
        hop = _smeared(U, dims, case["rho"], e.shift)
        e.H = [[hop[e.sites[p], mu].permute(1, 2, 0).contiguous() for mu in range(4)] for p in (0, 1)]
        psi = _in(_spinor(dims, seed, 0, True))
        return {"logdet": np.array([e.logdet]), "links": hop, "mhat": _native(e.mhat(psi, False), "single")}
    e = _Exact(case, dims, seed)
    psi = _in(_spinor(dims, seed, 0, prec != "double"))
    if kind == "apply":
        return _native(e.mdagm(psi), prec)
    if kind == "canonical":
        return e.mhat(psi, case["dagger"]).permute(2, 0, 1).contiguous()
    if kind == "solve":
        return e.solve(psi).permute(2, 0, 1).contiguous()
    return [e.solve(psi, s).permute(2, 0, 1).contiguous() for s in _SHIFTS]
