"""chi~0 over several panels of pairs: spheres with more pairs than a panel holds (terms of a pair and of its mirror image fall
into different panels), frequencies within one image of weights and beyond it; and systems of many transitions.

Bound per entry relative to the sum of the magnitudes of its terms: the weights, a and T are rounded to FP32 (5 x 2^-24), the
split products are within 2^-21, each chunk of 64 adds at most 12 truncations of 2^-23 and the promotion 2^-24 per
chunk; the terms of an entry are added in FP32, one rounding each.
"""
import numpy as np
import pytest

from synth import SystemSpec

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def bse():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as ge
    ge.build()
    from paper_1206_3518_gb300 import bse as b
    return b


def _dev(x, dtype):
    return torch.as_tensor(np.ascontiguousarray(x)).to(device="cuda", dtype=dtype)


@pytest.mark.parametrize("n,nv,nc,ecut,grid,nw", [(2, 1, 1, 12.0, 48, 40), (2, 1, 1, 12.0, 48, 1100), (6, 3, 4, 8.6, 32, 70),
                                                  (6, 3, 4, 8.6, 32, 1030)])
def test_several_panels(bse, n, nv, nc, ecut, grid, nw):
    spec = SystemSpec("cell", "fcc", 10.0, 0.0, (n, n, n), nv, nc, ecut, (grid,) * 3, "3d")
    plan = bse.Plan([spec])
    inf = plan.info(0)
    dim, ng = inf["dim"], inf["ng0"]
    kc = (dim + 63) // 64
    panel = (1 << 29) // ((kc * 512 + 4096) * 128) * 128
    assert ng * (ng + 1) // 2 > panel                    # more than one panel
    g = bse.bse_gvectors(plan, 0, 0, True)
    lut = {tuple(v): i for i, v in enumerate(g)}
    minus = np.array([lut[tuple(-v)] for v in g])
    rng = np.random.default_rng(7)
    rho = np.zeros((dim, inf["ng_max"]), dtype=np.complex64)
    rho[:, :ng] = (rng.standard_normal((dim, ng)) + 1j * rng.standard_normal((dim, ng))) * 10.0 ** rng.uniform(-3, 1, (1, ng))
    P = rng.standard_normal(dim) + 1j * rng.standard_normal(dim)
    en = np.sort(rng.uniform(-0.2, 0.0, (inf["nkpt"], nv)), axis=1)
    en = np.concatenate([en, np.sort(rng.uniform(0.05, 0.4, (inf["nkpt"], nc)), axis=1)], axis=1)
    omega, eta = np.linspace(0.0, 0.4, nw), 2e-3
    chi = torch.full((nw, ng, ng), float("nan"), dtype=torch.complex64, device="cuda")
    ws = torch.empty(bse.bse_workspace_size(plan, 0, bse.BSE_WS_CHI0) // 8 + 1, dtype=torch.complex64, device="cuda")
    bse.bse_chi0_optical(plan, 0, _dev(rho, torch.complex64), _dev(P, torch.complex128), _dev(en, torch.float64), 0.03,
                         _dev(omega, torch.float64), eta, chi, ws)
    bse.bse_status_read(plan)
    assert bool(torch.isfinite(torch.view_as_real(chi)).all())
    b = 2.0 * np.pi / 10.0 * np.array([[-1.0, 1, 1], [1, -1, 1], [1, 1, -1]])
    norm = np.linalg.norm(g @ b, axis=1)
    vh = np.sqrt(4.0 * np.pi) / np.where(norm > 0, norm, 1.0)
    r = rho[:, :ng].astype(np.complex128)
    a, ab = r * vh, r[:, minus].conj() * vh
    a[:, 0], ab[:, 0] = np.sqrt(4.0 * np.pi) * P.conj(), -np.sqrt(4.0 * np.pi) * P
    a, ab = torch.as_tensor(a, device="cuda"), torch.as_tensor(ab, device="cuda")
    de = torch.as_tensor((en[:, None, nv:] + 0.03 - en[:, :nv, None]).reshape(-1), device="cuda")
    tol = 6 * 2.0 ** -24 + 2.0 ** -21 + 12 * 2.0 ** -23 + kc * 2.0 ** -24
    for w in sorted({0, 31, 32, nw // 2, min(nw - 1, 127), min(nw - 1, 1023), nw - 1}):
        z = omega[w] + 1j * eta
        x, y = 1.0 / (z - de), -1.0 / (z + de)
        ref = 2.0 * inf["norm"] * ((a * x[:, None]).T @ a.conj() + (ab * y[:, None]).T @ ab.conj())
        size = 4.0 * inf["norm"] * ((a * x[:, None]).abs().T @ a.abs() + (ab * y[:, None]).abs().T @ ab.abs())
        assert bool(((chi[w].to(torch.complex128) - ref).abs() <= tol * size).all()), w
