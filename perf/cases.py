"""Performance cases of the Bethe-Salpeter path: the calls a user's program makes, over the range of sizes.

A case is one public entry point (or the ``Forward`` sequence of entry points) at one system size:

  build      H from coefficients, energies and W: ``Forward.build`` (pair densities, K^x, K^d)
  spectrum   eps_2 by the Haydock recursion on a given H (``bse_spectrum``)
  batch      eps_2 of several systems in one launch (``bse_spectrum_batch``)
  gradient   the adjoint of a spectral loss (``bse_spectrum_backward``)
  screening  the static RPA W of a q range from the states (BSE_PD_CHI0 + ``bse_screening``)
  chi0       the optical-limit response of TDDFT with local fields (``bse_chi0_optical``)
  dyson      its Dyson equation, eps_M(w) (``bse_epsilon_macro``)

Inputs are made on the device from the seed alone: random orthonormal plane-wave states, random band
energies and the model W of the synthetic workloads; the calls that take library-made intermediates
(H, pair densities, chi0) get random arrays of the same size, decay and spectrum.
"""
import itertools
import math
import random
from types import SimpleNamespace

import numpy as np
import torch

from paper_1206_3518_gb300 import bse
from paper_1206_3518_gb300.pipeline import Forward

EV = 1.0 / 27.211386245988
DEV = "cuda"
C64, C128 = torch.complex64, torch.complex128
HEX_A, HEX_C, HEX_ECUT, HEX_R0 = 4.7, 30.0, 2.5, 25.0   # the layered sheets of the batch workload
GAP_FLOOR = 0.1 * EV


def listed():
    fcc8 = {"lattice": "fcc", "n": 8, "nv": 3, "nc": 4, "ecut": 8.6, "grid": 32}
    return [
        # the small bulk cell of the tests: launches and latency are most of a build
        {"name": "build_fcc4_3v3c", "kind": "build", "lattice": "fcc", "n": 4, "nv": 3, "nc": 3, "ecut": 4.0,
         "grid": 24, "prec": "fp32", "qchunk": 64},
        # one layered sheet: odd mesh, slab Coulomb, small spheres, ragged tiles
        {"name": "build_sheet27_2v3c", "kind": "build", "lattice": "hex", "n": 27, "nv": 2, "nc": 3, "ecut": HEX_ECUT,
         "grid": 12, "prec": "fp32", "qchunk": 64},
        # the ordinary bulk calculation at the default precision
        {"name": "build_fcc8_3v4c", "kind": "build", **fcc8, "prec": "fp32", "qchunk": 512},
        # the same in the mixed precision
        {"name": "build_fcc8_3v4c_mixed", "kind": "build", **fcc8, "prec": "bf16x3", "qchunk": 512},
        # the largest bulk calculation (dim 27648), streamed over whole planes of the q mesh
        {"name": "build_fcc12_4v4c_mixed", "kind": "build", "lattice": "fcc", "n": 12, "nv": 4, "nc": 4, "ecut": 12.0,
         "grid": 48, "prec": "bf16x3", "qchunk": 144},
        # spectra: the small cell, and the ordinary one
        {"name": "spectrum_576", "kind": "spectrum", "n": 4, "nv": 3, "nc": 3, "nsteps": 100, "nw": 1000},
        {"name": "spectrum_6144", "kind": "spectrum", "n": 8, "nv": 3, "nc": 4, "nsteps": 300, "nw": 2000},
        # spectra of a set of sheets of uneven size in one launch
        {"name": "spectrum_6_sheets", "kind": "batch", "sheets": 6, "mix": 1, "nsteps": 300, "nw": 2000},
        # inverse problems: the gradient of a loss with respect to Delta, H, the pair densities and W
        {"name": "gradient_fcc8_3v4c", "kind": "gradient", **fcc8, "nsteps": 300, "nw": 512},
        # W from the system's own states, streamed over q
        {"name": "screening_fcc8_64q", "kind": "screening", **fcc8, "q0": 0, "nq": 64, "iterations": 16},
        # TDDFT with local fields: the response, and the Dyson equation with a kernel F
        {"name": "chi0_fcc8_1000w", "kind": "chi0", **fcc8, "nw": 1000},
        {"name": "dyson_fcc8_2000w", "kind": "dyson", **fcc8, "nw": 2000, "xc": True},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _bulk(rng, n):
    """A bulk system of n^3 k points: cutoff, bands, and the smallest real-space grid compiled for both."""
    nv, nc = rng.choice([(2, 2), (3, 3), (3, 4), (4, 4), (1, 2)])
    case = {"lattice": "fcc", "n": n, "nv": nv, "nc": nc, "ecut": round(rng.uniform(3.0, 10.0), 2)}
    g = np.concatenate(Geometry(case).g)
    reach = int(max(g.max() + 1, -g.min()))            # pair densities are taken at G - G0, G0 in {-1, 0}
    if reach <= 3 and nc <= 3:
        return {**case, "grid": 24}
    if reach <= 5 and nv + nc <= 7:
        return {**case, "grid": 32}
    return {**case, "grid": 48} if reach <= 6 else _bulk(rng, n)


def draw(rng):
    kind = rng.choice(["build", "build", "build", "sheet", "spectrum", "batch", "gradient", "screening", "chi0", "dyson"])
    n = rng.randint(3, 7 if kind == "gradient" else 8)
    bulk = _bulk(rng, n)
    if kind == "build":
        # q chunks as a user bounds memory: everything at once, or a few planes of the mesh
        return {"kind": "build", **bulk, "prec": rng.choice(["fp32", "bf16x3"]),
                "qchunk": rng.choice([n ** 3, n * n, 2 * n * n])}
    if kind == "sheet":
        return {"kind": "build", "lattice": "hex", "n": rng.randint(18, 32), "nv": rng.randint(1, 3),
                "nc": rng.randint(1, 3), "ecut": HEX_ECUT, "grid": 12, "prec": rng.choice(["fp32", "fp32", "bf16x3"]),
                "qchunk": 64}
    if kind == "spectrum":
        return {"kind": "spectrum", "n": rng.randint(3, 10), "nv": bulk["nv"], "nc": bulk["nc"],
                "nsteps": _log_int(rng, 40, 300), "nw": _log_int(rng, 200, 2000)}
    if kind == "batch":
        return {"kind": "batch", "sheets": rng.randint(2, 8), "mix": rng.randint(2, 10 ** 6),
                "nsteps": _log_int(rng, 40, 300), "nw": _log_int(rng, 200, 2000)}
    if kind == "gradient":
        return {"kind": "gradient", **bulk, "nsteps": _log_int(rng, 40, 300), "nw": _log_int(rng, 64, 1000)}
    if kind == "screening":
        nq = _log_int(rng, 2, min(64, n ** 3))
        return {"kind": "screening", **bulk, "q0": rng.randint(0, n ** 3 - nq), "nq": nq, "iterations": 16}
    if kind == "chi0":
        return {"kind": "chi0", **bulk, "nw": _log_int(rng, 50, 1000)}
    return {"kind": "dyson", **bulk, "nw": _log_int(rng, 50, 2000), "xc": rng.random() < 0.5}


# ---------------------------------------------------------------------------- geometry (numpy)

class Geometry:
    """Lattice, meshes, plane-wave spheres in the library's canonical order, and (k, k') blocks."""

    def __init__(self, case):
        n, a = case["n"], 10.0 if case["lattice"] == "fcc" else HEX_A
        self.fcc = case["lattice"] == "fcc"
        self.nv, self.nc, self.ecut = case["nv"], case["nc"], case["ecut"]
        self.nk = (n, n, n) if self.fcc else (n, n, 1)
        self.A = (0.5 * a * np.array([[0., 1, 1], [1, 0, 1], [1, 1, 0]]) if self.fcc else
                  np.array([[a, 0, 0], [-0.5 * a, 0.5 * math.sqrt(3.0) * a, 0], [0, 0, HEX_C]]))
        self.B = 2.0 * math.pi * np.linalg.inv(self.A).T
        self.omega = abs(np.linalg.det(self.A))
        self.nkpt = int(np.prod(self.nk))
        self.dim = self.nkpt * self.nv * self.nc
        self.norm = 1.0 / (self.omega * self.nkpt)
        self.k = np.array(list(itertools.product(*[range(m) for m in self.nk])), dtype=np.int64)
        r = math.sqrt(2.0 * self.ecut)
        m = [int(r * np.linalg.norm(v) / (2.0 * math.pi)) + 2 for v in self.A]
        box = np.array(list(itertools.product(*[range(-x, x + 1) for x in m])), dtype=np.int64)
        self.g, self.p2 = [], []
        for off in self.k:
            key, rhs, p2 = self._key(box, off, a)
            t = np.nonzero(key <= rhs)[0]
            t = t[np.lexsort((box[t, 2], box[t, 1], box[t, 0], key[t]))]
            self.g.append(box[t])
            self.p2.append(p2[t])
        self.ng = np.array([len(g) for g in self.g])
        self.ng_max = int(self.ng.max())

    def _key(self, g, off, a):
        n = self.nk[0]
        if self.fcc:
            x = n * g + off
            q = 3 * (x * x).sum(1) - 2 * (x[:, 0] * x[:, 1] + x[:, 0] * x[:, 2] + x[:, 1] * x[:, 2])
            t = a / (2.0 * math.pi)
            key = q.astype(float)
            return key, 2.0 * self.ecut * (t * t) * float(n * n), key * (2.0 * math.pi / a) ** 2 / (n * n)
        x, y = n * g[:, 0] + off[0], n * g[:, 1] + off[1]
        s, u = 2.0 * math.pi / a, 2.0 * math.pi / HEX_C
        z = (n * g[:, 2]).astype(float)
        key = (4.0 / 3.0) * (s * s) * (x * x + x * y + y * y).astype(float) + (u * u) * (z * z)
        return key, 2.0 * self.ecut * float(n * n), key / (n * n)

    def cart(self, ik, g):
        return (g + self.k[ik] / np.array(self.nk)) @ self.B

    def v_half(self, iq):
        """sqrt of the Coulomb interaction on the sphere of q (0 at q + G = 0), and |(q + G)_parallel|."""
        p = self.cart(iq, self.g[iq])
        par, p2 = np.linalg.norm(p[:, :2], axis=1), self.p2[iq]
        with np.errstate(divide="ignore", invalid="ignore"):
            v = 4.0 * math.pi / p2
            if not self.fcc:
                v = v * (1.0 - np.exp(-par * 0.5 * HEX_C) * np.cos(0.5 * HEX_C * p[:, 2]))
        return np.sqrt(np.where(p2 > 0, np.maximum(v, 0.0), 0.0)), par

    def head(self):
        if self.fcc:
            qc = (6.0 * math.pi ** 2 / (self.omega * self.nkpt)) ** (1.0 / 3.0)
            return 12.0 * math.pi / (qc * qc)
        area = abs(np.linalg.det(self.A[:2, :2]))
        qc = math.sqrt(4.0 * math.pi / (area * self.nkpt))
        q = (np.arange(64) + 0.5) / 64 * qc
        f = 2.0 * math.pi * q * 4.0 * math.pi * (1.0 - np.exp(-0.5 * q * HEX_C)) / (q * q) / (1.0 + HEX_R0 * q)
        return float(f.mean() * qc / (math.pi * qc * qc))

    def lin(self, i):
        return (i[..., 0] * self.nk[1] + i[..., 1]) * self.nk[2] + i[..., 2]

    def blocks(self, iq):
        """Upper blocks (k, k') of q and their G0: k' = fold(k + q) >= k, G0 = (k' - k - q)/n."""
        s = self.k + self.k[iq]
        f = s % np.array(self.nk)
        ik2 = self.lin(f)
        t = np.nonzero(np.arange(self.nkpt) <= ik2)[0]
        return t, ik2[t], ((f - s) // np.array(self.nk))[t]


def _plan(case, geo):
    spec = SimpleNamespace(lattice=case["lattice"], a=10.0 if geo.fcc else HEX_A, c=0.0 if geo.fcc else HEX_C,
                           nk=geo.nk, nv=geo.nv, nc=geo.nc, ecut=geo.ecut,
                           fft=(case["grid"],) * 3 if geo.fcc else (12, 12, 48), coulomb="3d" if geo.fcc else "slab")
    return bse.Plan([spec])


# ---------------------------------------------------------------------------- inputs (torch, from the seed)

def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _cplx(gen, *shape, dtype=C64):
    re = torch.float32 if dtype == C64 else torch.float64
    return torch.view_as_complex(torch.randn(*shape, 2, generator=gen, device=DEV, dtype=re)) * (0.5 ** 0.5)


def _padded(rows, width):
    out = np.zeros((len(rows), width))
    for i, r in enumerate(rows):
        out[i, : len(r)] = r
    return torch.as_tensor(out, device=DEV)


def _mask(geo):
    return torch.arange(geo.ng_max, device=DEV)[None, :] < torch.as_tensor(geo.ng, device=DEV)[:, None]


def _states(geo, gen):
    """Orthonormal random states with Gaussian decay (coefficients [k][band][G]) and sorted random energies."""
    nb = geo.nv + geo.nc
    amp = torch.exp(-_padded(geo.p2, geo.ng_max) / 8.0) * _mask(geo)
    z = _cplx(gen, geo.nkpt, geo.ng_max, nb, dtype=C128) * amp[:, :, None]
    chol = torch.linalg.cholesky(z.mH @ z)
    q = torch.linalg.solve_triangular(chol, z.mT.conj(), upper=False)     # rows: orthonormal bands, conjugated
    return q.conj().to(C64).contiguous(), _energies(geo, gen)


def _energies(geo, gen):
    u = torch.rand(geo.nkpt, geo.nv + geo.nc, generator=gen, device=DEV, dtype=torch.float64)
    ev = torch.sort(-6.0 + 6.0 * u[:, : geo.nv], dim=1).values
    ec = torch.sort(1.5 + 8.5 * u[:, geo.nv:], dim=1).values
    return (torch.cat([ev, ec], dim=1) * EV).contiguous()


def _w_model(geo, gen):
    """W_q = v^1/2 eps^-1 v^1/2 with the model eps^-1 (diagonal decay, small random Hermitian part)."""
    W = torch.zeros(geo.nkpt, geo.ng_max, geo.ng_max, dtype=C64, device=DEV)
    vh, par = zip(*[geo.v_half(iq) for iq in range(geo.nkpt)])
    vh, par, p2 = _padded(vh, geo.ng_max), _padded(par, geo.ng_max), _padded(geo.p2, geo.ng_max)
    d = 1.0 - (1.0 - 1.0 / 11.0) * torch.exp(-p2 / 4.0) if geo.fcc else 1.0 / (1.0 + HEX_R0 * par)
    vh = (vh * _mask(geo)).float()
    amp = vh * d.float().sqrt() * (0.02 ** 0.5 / geo.ng_max ** 0.25)
    step = max(1, (1 << 26) // geo.ng_max ** 2)
    for a in range(0, geo.nkpt, step):
        b = min(a + step, geo.nkpt)
        h = torch.triu(_cplx(gen, b - a, geo.ng_max, geo.ng_max), 1)
        h = (h + h.mH) * (amp[a:b, :, None] * amp[a:b, None, :])
        W[a:b] = h + torch.diag_embed((vh[a:b] ** 2 * d[a:b].float()).to(C64))
    W[0, 0, :] = 0.0
    W[0, :, 0] = 0.0
    W[0, 0, 0] = geo.head() / (11.0 if geo.fcc else 1.0)
    return W


def _hamiltonian(dim, gen):
    """Transition energies on the diagonal, a small random Hermitian coupling off it."""
    H = _cplx(gen, dim, dim)
    H = (H + H.mH) * (0.03 / math.sqrt(dim))
    de = (2.0 + 14.0 * torch.rand(dim, generator=gen, device=DEV)) * EV
    H.diagonal().copy_(de.to(C64))
    return H


def _densities(geo, gen, rows, p2):
    """Random pair densities [rows][ng_max] decaying with |q + G|."""
    amp = 0.1 * torch.exp(-torch.as_tensor(p2, device=DEV) / 12.0).float()
    out = torch.zeros(rows, geo.ng_max, dtype=C64, device=DEV)
    out[:, : len(p2)] = _cplx(gen, rows, len(p2)) * amp
    return out


def _omega(nw):
    return torch.linspace(0.0, 10.0 * EV, nw, dtype=torch.float64, device=DEV)


def _spectrum_geo(case):
    return {"lattice": "fcc", "ecut": 4.0, "grid": 24, **case}


def _sheet_cases(case):
    """n x n sheets of uneven size and bands, the first of them large."""
    rng = random.Random(case["mix"])
    sizes = [(rng.randint(18, 36), rng.randint(1, 2), rng.randint(1, 3)) for _ in range(case["sheets"])]
    return [{"lattice": "hex", "n": n, "nv": v, "nc": c, "ecut": HEX_ECUT, "grid": 12} for n, v, c in sizes]


def _nvec(geo):
    return geo.nkpt * (geo.nkpt + 1) // 2 * (geo.nv ** 2 + geo.nc ** 2)


def _workspace(plan, s, kind, arg):
    return torch.empty(bse.bse_workspace_size(plan, s, kind, arg) // 8 + 1, dtype=C64, device=DEV)


class _Spectrum:
    """Buffers of one system's spectrum."""

    def __init__(self, plan, s, dim, case, gen):
        self.H = _hamiltonian(dim, gen)
        self.P = _cplx(gen, dim, dtype=C128)
        self.eps2 = torch.zeros(case["nw"], dtype=torch.float64, device=DEV)
        self.ab = torch.zeros(2 * case["nsteps"], dtype=torch.float64, device=DEV)
        self.done = torch.zeros(1, dtype=torch.int32, device=DEV)
        self.ws = _workspace(plan, s, bse.BSE_WS_SPECTRUM, case["nsteps"])

    def outputs(self):
        return {"eps2": self.eps2, "ab": self.ab, "steps": self.done}


def _inputs(case, seed):
    """The arrays of a case that do not come from the library (shared with exact())."""
    gen, kind = _gen(seed), case["kind"]
    st = SimpleNamespace(case=case)
    if kind == "build":
        st.geo = Geometry(case)
        st.coef, st.en = _states(st.geo, gen)
        st.W = _w_model(st.geo, gen)
    elif kind == "gradient":
        st.geo = geo = Geometry(case)
        st.H, st.P = _hamiltonian(geo.dim, gen), _cplx(gen, geo.dim, dtype=C128)
        st.rho_x = _densities(geo, gen, geo.dim, geo.p2[0])
        st.rho_dir = torch.cat([_densities(geo, gen, len(geo.blocks(iq)[0]) * (geo.nv ** 2 + geo.nc ** 2), geo.p2[iq])
                                for iq in range(geo.nkpt)])
        st.W = _w_model(geo, gen)
        st.g = torch.randn(case["nw"], generator=gen, device=DEV, dtype=torch.float64) / case["nw"]
    elif kind == "screening":
        st.geo = Geometry(case)
        st.coef, st.en = _states(st.geo, gen)
        st.P = _cplx(gen, st.geo.dim, dtype=C128)
    elif kind == "chi0":
        st.geo = Geometry(case)
        st.rho_x = _densities(st.geo, gen, st.geo.dim, st.geo.p2[0])
        st.P = 0.3 * _cplx(gen, st.geo.dim, dtype=C128)
        st.en = _energies(st.geo, gen)
    elif kind == "dyson":
        st.geo = geo = Geometry(case)
        ng = int(geo.ng[0])
        amp = torch.exp(-torch.as_tensor(geo.p2[0], device=DEV) / 8.0).float()
        st.chi = _cplx(gen, case["nw"], ng, ng) * (0.2 / math.sqrt(ng)) * (amp[:, None] * amp[None, :])
        st.chi.diagonal(dim1=1, dim2=2).sub_(0.8 * amp ** 2)
        st.F = None
        if case["xc"]:
            f = torch.triu(_cplx(gen, ng, ng), 1) * 0.01
            st.F = (f + f.mH - 0.1 * torch.eye(ng, device=DEV)).contiguous()
    return st


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("spectrum", "batch"):
        gen = _gen(seed)
        geos = [Geometry(c) for c in ([_spectrum_geo(case)] if kind == "spectrum" else _sheet_cases(case))]
        cases = [_spectrum_geo(case)] if kind == "spectrum" else _sheet_cases(case)
        specs = [SimpleNamespace(lattice=c["lattice"], a=10.0 if g.fcc else HEX_A, c=0.0 if g.fcc else HEX_C, nk=g.nk,
                                 nv=g.nv, nc=g.nc, ecut=g.ecut, fft=(24, 24, 24) if g.fcc else (12, 12, 48),
                                 coulomb="3d" if g.fcc else "slab") for c, g in zip(cases, geos)]
        plan = bse.Plan(specs)
        return SimpleNamespace(case=case, plan=plan, omega=_omega(case["nw"]),
                               sys=[_Spectrum(plan, i, g.dim, case, gen) for i, g in enumerate(geos)])
    st = _inputs(case, seed)
    geo = st.geo
    st.plan = plan = _plan(case, geo)
    if kind == "build":
        st.F = Forward(plan, 0, nsteps=1, nw=1, qchunk=min(case["qchunk"], geo.nkpt))
        st.prec = bse.BSE_PREC_FP32 if case["prec"] == "fp32" else bse.BSE_PREC_BF16X3
    elif kind == "gradient":
        st.omega = _omega(case["nw"])
        st.ws = _workspace(plan, 0, bse.BSE_WS_BACKWARD, case["nsteps"])
        st.out = {"ddelta": torch.zeros(1, dtype=torch.float64, device=DEV), "dH": torch.zeros_like(st.H),
                  "drho_x": torch.zeros_like(st.rho_x), "drho_dir": torch.zeros_like(st.rho_dir),
                  "dW": torch.zeros_like(st.W)}
    elif kind == "screening":
        nq = case["nq"]
        st.ws_pair = _workspace(plan, 0, bse.BSE_WS_PAIR, 0)
        st.ws = _workspace(plan, 0, bse.BSE_WS_SCREEN, nq)
        st.rho = torch.zeros(nq * geo.dim, geo.ng_max, dtype=C64, device=DEV)
        st.W = torch.zeros(geo.nkpt, geo.ng_max, geo.ng_max, dtype=C64, device=DEV)
        bse.bse_pair_densities(plan, 0, bse.BSE_PD_REALSPACE, st.coef, st.en, None, None, None, 0, 0, st.ws_pair)
    elif kind == "chi0":
        ng = int(geo.ng[0])
        st.omega = _omega(case["nw"])
        st.ws = _workspace(plan, 0, bse.BSE_WS_CHI0, 0)
        st.chi = torch.empty(case["nw"], ng, ng, dtype=C64, device=DEV)
    elif kind == "dyson":
        st.ws = _workspace(plan, 0, bse.BSE_WS_EPSM, case["nw"])
        st.eps_m = torch.zeros(case["nw"], dtype=C128, device=DEV)
    return st


def run(st):
    case, kind, plan = st.case, st.case["kind"], st.plan
    if kind == "build":
        return {"H": st.F.build(st.coef, st.en, st.W, 0.8 * EV, st.prec), "P": st.F.P}
    if kind == "spectrum":
        s = st.sys[0]
        bse.bse_spectrum(plan, 0, s.H, s.P, case["nsteps"], st.omega, 0.05 * EV, s.eps2, s.ab, s.done, s.ws)
        return s.outputs()
    if kind == "batch":
        S = st.sys
        bse.bse_spectrum_batch(plan, list(range(len(S))), [s.H for s in S], [s.P for s in S], case["nsteps"], st.omega,
                               0.05 * EV, [s.eps2 for s in S], [s.ab for s in S], [s.done for s in S], [s.ws for s in S])
        return [s.outputs() for s in S]
    if kind == "gradient":
        o = st.out
        bse.bse_spectrum_backward(plan, 0, st.H, st.P, case["nsteps"], st.omega, 0.05 * EV, st.g, st.rho_x, st.rho_dir,
                                  st.W, o["ddelta"], o["dH"], o["drho_x"], o["drho_dir"], o["dW"], st.ws)
        return o
    if kind == "screening":
        q0, q1 = case["q0"], case["q0"] + case["nq"]
        bse.bse_pair_densities(plan, 0, bse.BSE_PD_CHI0, None, None, None, None, st.rho, q0, q1, st.ws_pair)
        bse.bse_screening(plan, 0, st.rho, st.en, st.P, q0, q1, case["iterations"], st.W, None, st.ws)
        return st.W[q0:q1]
    if kind == "chi0":
        bse.bse_chi0_optical(plan, 0, st.rho_x, st.P, st.en, 0.8 * EV, st.omega, 0.05 * EV, st.chi, st.ws)
        return st.chi
    bse.bse_epsilon_macro(plan, 0, st.chi, st.F, st.eps_m, st.ws)
    return st.eps_m


# ---------------------------------------------------------------------------- necessary work

def work(case):
    kind = case["kind"]
    if kind in ("spectrum", "batch"):
        dims = ([case["n"] ** 3 * case["nv"] * case["nc"]] if kind == "spectrum" else
                [c["n"] ** 2 * c["nv"] * c["nc"] for c in _sheet_cases(case)])
        n = case["nsteps"]
        # every step reads H once; products with H, and two Gram-Schmidt passes over the basis
        return {"bytes": sum(8.0 * n * d * d + 16.0 * d for d in dims),
                "flops": sum(8.0 * n * d * d + 16.0 * n * n * d for d in dims)}
    geo = Geometry(case)
    ng, nb = float(geo.ng_max), geo.nv + geo.nc
    v2, c2, nblk = geo.nv ** 2, geo.nc ** 2, geo.nkpt * (geo.nkpt + 1) / 2.0
    W, H = 8.0 * geo.nkpt * ng * ng, 8.0 * float(geo.dim) ** 2
    if kind == "build":
        return {"bytes": 8.0 * geo.nkpt * nb * (ng + 1) + W + H,
                "flops": 8.0 * nblk * ((v2 + c2) * ng * ng + min(v2, c2) * ng * ng + v2 * c2 * ng) + 4.0 * geo.dim ** 2 * ng}
    if kind == "gradient":
        n = case["nsteps"]
        return {"bytes": 8.0 * n * geo.dim ** 2 + 2 * W + 2 * H + 16.0 * _nvec(geo) * ng + 16.0 * geo.dim * ng,
                "flops": 8.0 * n * geo.dim ** 2 + 16.0 * n * n * geo.dim + 4.0 * n * geo.dim ** 2 + 8.0 * geo.dim ** 2 * ng
                + 8.0 * nblk * ((v2 + 2 * c2) * ng * ng + 3 * v2 * c2 * ng)}
    if kind == "screening":
        nq = case["nq"]
        return {"bytes": 8.0 * geo.nkpt * nb * ng + 8.0 * nq * ng * ng,
                "flops": 8.0 * nq * (geo.dim * ng * ng + 0.5 * geo.dim * ng * ng + ng ** 3)}
    n0 = float(geo.ng[0])
    if kind == "chi0":
        return {"bytes": 8.0 * geo.dim * n0 + 8.0 * case["nw"] * n0 * n0, "flops": 8.0 * case["nw"] * geo.dim * n0 * n0}
    return {"bytes": 8.0 * case["nw"] * n0 * n0, "flops": case["nw"] * n0 ** 3 * (8.0 / 3.0 + (8.0 if case["xc"] else 0.0))}


# ---------------------------------------------------------------------------- 64-bit references (torch, complex128)

def _box(geo, ik, reach):
    """Dense table (G1 + reach) -> index on the sphere of k, ng_max outside it."""
    dims = [2 * r + 1 for r in reach]
    t = torch.full((dims[0] * dims[1] * dims[2],), geo.ng_max, dtype=torch.int64, device=DEV)
    g = torch.as_tensor(geo.g[ik] + np.array(reach), device=DEV)
    t[(g[:, 0] * dims[1] + g[:, 1]) * dims[2] + g[:, 2]] = torch.arange(len(g), device=DEV)
    return t, dims


class _Correlator:
    """rho_nm(G) = sum_{G2 in S(k')} conj(c_nk(G2 - G)) c_mk'(G2) in 64 bits for a batch of k' at one k."""

    def __init__(self, geo, coef):
        self.geo, self.c = geo, coef.to(C128)
        fmax = np.abs(np.concatenate(geo.g)).max(0)
        self.reach = [int(2 * f + 1) for f in fmax]
        self.g = torch.zeros(geo.nkpt, geo.ng_max, 3, dtype=torch.int64, device=DEV)
        for ik in range(geo.nkpt):
            self.g[ik, : geo.ng[ik]] = torch.as_tensor(geo.g[ik], device=DEV)

    def __call__(self, ik, ik2, iq, g0, left, right):
        """[batch][left band][right band][G] at G = g_p(q) - G0, zero beyond the sphere of q."""
        geo, reach = self.geo, self.reach
        table, dims = _box(geo, ik, reach)
        G = self.g[iq] - torch.as_tensor(g0, device=DEV)[:, None, :]
        d = self.g[ik2][:, None, :, :] - G[:, :, None, :] + torch.tensor(reach, device=DEV)
        idx = table[(d[..., 0] * dims[1] + d[..., 1]) * dims[2] + d[..., 2]]       # [batch][G][G2]
        cl = torch.cat([self.c[ik, left], torch.zeros(len(left), 1, dtype=C128, device=DEV)], dim=1).conj()
        cr = self.c[ik2][:, right]
        out = torch.einsum("nbgh,bmh->bnmg", cl[:, idx], cr)
        keep = torch.arange(geo.ng_max, device=DEV)[None, :] < torch.as_tensor(geo.ng, device=DEV)[iq][:, None]
        return out * keep[:, None, None, :]


def _exact_dipole(geo, coef, en):
    c, P = coef.to(C128), torch.zeros(geo.nkpt, geo.nv, geo.nc, dtype=C128, device=DEV)
    kx = torch.zeros(geo.nkpt, geo.ng_max, dtype=torch.float64, device=DEV)
    for ik in range(geo.nkpt):
        kx[ik, : geo.ng[ik]] = torch.as_tensor(geo.cart(ik, geo.g[ik])[:, 0], device=DEV)
    m = torch.einsum("kvg,kg,kcg->kvc", c[:, : geo.nv].conj(), kx.to(C128), c[:, geo.nv:])
    P = m.conj() / (en[:, None, geo.nv:] - en[:, : geo.nv, None]).clamp_min(GAP_FLOOR)
    return P.reshape(-1)


def _exact_build(st):
    geo, nv, nc = st.geo, st.geo.nv, st.geo.nc
    nvc, V, Cb = nv * nc, list(range(nv)), list(range(nv, nv + nc))
    corr = _Correlator(geo, st.coef)
    vh = torch.as_tensor(geo.v_half(0)[0], device=DEV)
    zero = np.zeros((1, 3), dtype=np.int64)
    rx = torch.cat([corr(k, [k], [0], zero, V, Cb).reshape(nvc, -1) for k in range(geo.nkpt)])[:, : geo.ng[0]]
    y = rx * (vh * math.sqrt(2.0 * geo.norm))
    H = (y.conj() @ y.T).reshape(geo.nkpt, nvc, geo.nkpt, nvc)
    W = st.W.to(C128)
    step = max(1, (1 << 28) // ((nv + nc) * geo.ng_max ** 2))
    for ik in range(geo.nkpt):
        for a in range(ik, geo.nkpt, step):
            k2 = np.arange(a, min(a + step, geo.nkpt))
            dk = geo.k[k2] - geo.k[ik]
            iq = geo.lin(dk % np.array(geo.nk))
            g0 = (dk - geo.k[iq]) // np.array(geo.nk)
            rv, rc = corr(ik, k2, iq, g0, V, V), corr(ik, k2, iq, g0, Cb, Cb)
            X = torch.einsum("bcdg,bhg->bcdh", rc, W[iq])
            M = torch.einsum("bvwg,bcdg->vcbwd", rv.conj(), X).reshape(nvc, len(k2), nvc)
            H[ik][:, k2] -= geo.norm * M
    H = H.reshape(geo.dim, geo.dim)
    de = (st.en[:, None, nv:] + 0.8 * EV - st.en[:, :nv, None]).reshape(-1)
    H += torch.diag(de).to(C128)
    up = torch.arange(geo.nkpt, device=DEV).repeat_interleave(nvc)
    low, same = up[:, None] > up[None, :], up[:, None] == up[None, :]
    Hh = H.mH
    return {"H": torch.where(low, Hh, torch.where(same, 0.5 * (H + Hh), H)), "P": _exact_dipole(geo, st.coef, st.en)}


def _lanczos(H, P, n):
    """Basis [n][dim], a, b of the Haydock recursion with full reorthogonalisation in 64 bits."""
    H = H.to(C128)
    V = torch.zeros(n, H.shape[0], dtype=C128, device=DEV)
    V[0] = P / torch.linalg.norm(P)
    a, b = np.zeros(n), np.zeros(n)
    for j in range(n):
        w = H @ V[j]
        for _ in range(2):
            h = V[: j + 1].conj() @ w
            a[j] += float(h[j].real)
            w = w - h @ V[: j + 1]
        if j + 1 < n:
            b[j + 1] = float(torch.linalg.norm(w))
            V[j + 1] = w / b[j + 1]
    return V, a, b


def _prefactor(geo):
    return 8.0 * math.pi / (geo.omega * geo.nkpt)


def _exact_spectrum(s, geo, case, omega):
    n, z = case["nsteps"], omega.cpu().numpy() + 0.05j * EV
    _, a, b = _lanczos(s.H, s.P, n)
    g = np.zeros_like(z)
    for j in range(n - 1, -1, -1):
        g = 1.0 / (z - a[j] - (b[j + 1] ** 2 * g if j + 1 < n else 0.0))
    eps2 = -_prefactor(geo) * float(torch.linalg.norm(s.P)) ** 2 * g.imag
    return {"eps2": eps2, "ab": np.concatenate([a, b]), "steps": None}


def _exact_gradient(st):
    geo, n, nv, nc = st.geo, st.case["nsteps"], st.geo.nv, st.geo.nc
    V, a, b = _lanczos(st.H, st.P, n)
    z = torch.as_tensor(_omega(st.case["nw"]).cpu().numpy() + 0.05j * EV, device=DEV)
    T = torch.as_tensor(np.diag(a) + np.diag(b[1:], 1) + np.diag(b[1:], -1), device=DEV).to(C128)
    e0 = torch.zeros(len(z), n, 1, dtype=C128, device=DEV)
    e0[:, 0] = 1.0
    y = torch.linalg.solve(z[:, None, None] * torch.eye(n, device=DEV, dtype=C128) - T, e0)[..., 0]
    p2 = float(torch.linalg.norm(st.P)) ** 2
    M = -_prefactor(geo) * p2 * ((y * st.g[:, None]).T @ y).imag
    G = V.T @ (M.to(C128) @ V.conj())
    vh = torch.zeros(geo.ng_max, dtype=torch.float64, device=DEV)
    vh[: geo.ng[0]] = torch.as_tensor(geo.v_half(0)[0], device=DEV)
    drx = 4.0 * geo.norm * vh ** 2 * (G.conj() @ st.rho_x.to(C128))
    drd, dW, at = torch.zeros(st.rho_dir.shape, dtype=C128, device=DEV), torch.zeros(st.W.shape, dtype=C128, device=DEV), 0
    G5 = G.reshape(geo.nkpt, nv, nc, geo.nkpt, nv, nc)
    for iq in range(geo.nkpt):
        k, k2, _ = geo.blocks(iq)
        ng, nb = int(geo.ng[iq]), len(k)
        fac = torch.as_tensor(np.where(k == k2, 1.0, 2.0), device=DEV)
        Gm = G5[k, :, :, k2] * fac[:, None, None, None, None]                       # [block][v][c][v'][c']
        nvv, ncc = nb * nv * nv, nb * nc * nc
        Rv = st.rho_dir[at: at + nvv, :ng].to(C128).reshape(nb, nv, nv, ng)
        Rc = st.rho_dir[at + nvv: at + nvv + ncc, :ng].to(C128).reshape(nb, nc, nc, ng)
        Wq = st.W[iq, :ng, :ng].to(C128)
        Xv, Xc = Rv @ Wq.T, Rc @ Wq.T
        drd[at: at + nvv, :ng] = -geo.norm * torch.einsum("bvcwd,bcdg->bvwg", Gm.conj(), Xc).reshape(nvv, ng)
        drd[at + nvv: at + nvv + ncc, :ng] = -geo.norm * torch.einsum("bvcwd,bvwg->bcdg", Gm, Xv).reshape(ncc, ng)
        Y = torch.einsum("bvcwd,bvwg->bcdg", Gm, Rv).reshape(ncc, ng)
        dW[iq, :ng, :ng] = -geo.norm * (Y.T @ Rc.reshape(ncc, ng).conj())
        at += nvv + ncc
    return {"ddelta": torch.trace(M).reshape(1), "dH": G, "drho_x": drx, "drho_dir": drd, "dW": dW}


def _exact_screening(st):
    geo, case, nv, nc = st.geo, st.case, st.geo.nv, st.geo.nc
    q0, nq, ng = case["q0"], case["nq"], geo.ng_max
    corr = _Correlator(geo, st.coef)
    V, Cb = list(range(nv)), list(range(nv, nv + nc))
    iqs = np.arange(q0, q0 + nq)
    vh = torch.stack([torch.cat([torch.as_tensor(geo.v_half(q)[0], device=DEV),
                                 torch.zeros(ng - geo.ng[q], dtype=torch.float64, device=DEV)]) for q in iqs])
    eps = torch.eye(ng, dtype=C128, device=DEV).repeat(nq, 1, 1)
    step = max(1, (1 << 28) // (nv * ng ** 2))
    for ik in range(geo.nkpt):
        for a in range(0, nq, step):
            t = iqs[a: a + step]
            s = geo.k[ik] + geo.k[t]
            f = s % np.array(geo.nk)
            k2 = geo.lin(f)
            r = corr(ik, k2, t, (f - s) // np.array(geo.nk), V, Cb)                 # [q][v][c][G]
            de = (st.en[k2][:, None, nv:] - st.en[ik, :nv][None, :, None]).clamp_min(GAP_FLOOR)
            w = torch.sqrt(4.0 * geo.norm / de)
            A = (r * w[..., None] * vh[a: a + len(t), None, None, :]).reshape(len(t), nv * nc, ng)
            if t[0] == 0:
                p = st.P[ik * nv * nc: (ik + 1) * nv * nc]
                A[0, :, 0] = p.conj() * math.sqrt(4.0 * math.pi) * w[0].reshape(-1)
            eps[a: a + len(t)] += A.mT @ A.conj()
    inv = torch.linalg.inv(eps)
    W = inv * (vh[:, :, None] * vh[:, None, :])
    if q0 == 0:
        W[0, 0, :] = 0.0
        W[0, :, 0] = 0.0
        W[0, 0, 0] = inv[0, 0, 0] * geo.head()
    return W


def _exact_chi0(st):
    geo, nv = st.geo, st.geo.nv
    ng, nw, dim = int(geo.ng[0]), st.case["nw"], geo.dim
    lut = {tuple(g): i for i, g in enumerate(geo.g[0])}
    minus = torch.as_tensor([lut[tuple(-g)] for g in geo.g[0]], device=DEV)
    vh = torch.as_tensor(geo.v_half(0)[0], device=DEV)
    r = st.rho_x[:, :ng].to(C128)
    a, ab = r * vh, r[:, minus].conj() * vh
    a[:, 0], ab[:, 0] = math.sqrt(4.0 * math.pi) * st.P.conj(), -math.sqrt(4.0 * math.pi) * st.P
    de = (st.en[:, None, nv:] + 0.8 * EV - st.en[:, :nv, None]).reshape(-1)
    z = _omega(nw).to(C128) + 0.05j * EV
    out = torch.empty(nw, ng, ng, dtype=C128, device=DEV)
    ah, abh = a.conj(), ab.conj()
    for w in range(nw):
        out[w] = (a / (z[w] - de)[:, None]).T @ ah - (ab / (z[w] + de)[:, None]).T @ abh
    return 2.0 * geo.norm * out


def _exact_dyson(st):
    ng, out = st.chi.shape[1], []
    eye = torch.eye(ng, dtype=C128, device=DEV)
    K = eye if st.F is None else eye + st.F.to(C128)
    for c in st.chi.split(250):
        c = c.to(C128)
        out.append(1.0 / (1.0 + torch.linalg.solve(eye - c @ K, c[:, :, :1])[:, 0, 0]))
    return torch.cat(out)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("build", "gradient", "screening") and work(case)["flops"] > 5e12:
        return None                      # over 20 s in 64 bits
    if kind in ("spectrum", "batch"):
        st = prepare(case, seed)
        geos = [Geometry(c) for c in ([_spectrum_geo(case)] if kind == "spectrum" else _sheet_cases(case))]
        out = [_exact_spectrum(s, g, case, st.omega) for s, g in zip(st.sys, geos)]
        return out[0] if kind == "spectrum" else out
    st = _inputs(case, seed)
    return {"build": _exact_build, "gradient": _exact_gradient, "screening": _exact_screening, "chi0": _exact_chi0,
            "dyson": _exact_dyson}[kind](st)
