"""Products of the TDDFT response and of the screening on the tensor cores, and the blocked Dyson elimination, at the
sizes where their tiles end: fewer transitions than a K chunk, frequencies on both sides of a 32-row tile of
weights and of a 128-frequency group, spheres below one panel and with a ragged last one, more q than one group.

Bound of chi~0 per entry, from the arithmetic, relative to the sum of the magnitudes of its terms: the weights, a and T are
rounded to FP32 (5 x 2^-24), the split products are within 2^-21, each chunk of 64 adds at most 12 truncations of 2^-23
and the promotion 2^-24 per chunk.
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


def _ws(bse, plan, kind, arg=0):
    return torch.empty(bse.bse_workspace_size(plan, 0, kind, arg) // 8 + 1, dtype=torch.complex64, device="cuda")


def _spec(n, nv, nc, ecut, grid):
    return SystemSpec("cell", "fcc", 10.0, 0.0, (n, n, n), nv, nc, ecut, (grid,) * 3, "3d")


@pytest.mark.parametrize("n,nv,nc,ecut,grid,nw", [(2, 1, 1, 1.0, 8, 1), (2, 2, 2, 1.0, 8, 31), (2, 2, 2, 1.0, 8, 33),
                                                  (3, 2, 2, 4.0, 24, 129), (2, 3, 4, 8.6, 32, 40)])
def test_chi0_of_random_densities(bse, n, nv, nc, ecut, grid, nw):
    spec = _spec(n, nv, nc, ecut, grid)
    plan = bse.Plan([spec])
    inf = plan.info(0)
    dim, ng = inf["dim"], inf["ng0"]
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
    bse.bse_chi0_optical(plan, 0, _dev(rho, torch.complex64), _dev(P, torch.complex128), _dev(en, torch.float64), 0.03,
                         _dev(omega, torch.float64), eta, chi, _ws(bse, plan, bse.BSE_WS_CHI0))
    bse.bse_status_read(plan)
    chi = chi.cpu().numpy()
    b = 2.0 * np.pi / 10.0 * np.array([[-1.0, 1, 1], [1, -1, 1], [1, 1, -1]])
    norm = np.linalg.norm(g @ b, axis=1)
    vh = np.sqrt(4.0 * np.pi) / np.where(norm > 0, norm, 1.0)
    r = rho[:, :ng].astype(np.complex128)
    a, ab = r * vh, r[:, minus].conj() * vh
    a[:, 0], ab[:, 0] = np.sqrt(4.0 * np.pi) * P.conj(), -np.sqrt(4.0 * np.pi) * P
    de = (en[:, None, nv:] + 0.03 - en[:, :nv, None]).reshape(-1)
    chunks = (dim + 63) // 64
    tol = 5 * 2.0 ** -24 + 2.0 ** -21 + 12 * 2.0 ** -23 + chunks * 2.0 ** -24
    for w in {0, nw // 2, nw - 1}:
        z = omega[w] + 1j * eta
        x, y = 1.0 / (z - de), -1.0 / (z + de)
        ref = 2.0 * inf["norm"] * ((a * x[:, None]).T @ a.conj() + (ab * y[:, None]).T @ ab.conj())
        size = 4.0 * inf["norm"] * (np.abs(a * x[:, None]).T @ np.abs(a) + np.abs(ab * y[:, None]).T @ np.abs(ab))
        assert np.all(np.abs(chi[w] - ref) <= tol * size), w


@pytest.mark.parametrize("n,ecut,grid,xc", [(2, 1.0, 8, True), (2, 1.6, 24, False), (2, 4.0, 24, True), (2, 8.6, 32, True),
                                            (2, 12.0, 48, False)])
def test_dyson_elimination(bse, n, ecut, grid, xc):
    """Random systems without diagonal dominance (rows are swapped in every panel) against the FP64 solution: elimination
    with partial pivoting is within ~8 n 2^-24 of the condition number."""
    spec = _spec(n, 1, 1, ecut, grid)
    plan = bse.Plan([spec])
    ng, nw = plan.info(0)["ng0"], 5
    rng = np.random.default_rng(3)
    chi = ((rng.standard_normal((nw, ng, ng)) + 1j * rng.standard_normal((nw, ng, ng))) * 0.7).astype(np.complex64)
    F = (0.05 * (rng.standard_normal((ng, ng)) + 1j * rng.standard_normal((ng, ng)))).astype(np.complex64) if xc else None
    eps = torch.zeros(nw, dtype=torch.complex128, device="cuda")
    bse.bse_epsilon_macro(plan, 0, _dev(chi, torch.complex64), None if F is None else _dev(F, torch.complex64), eps,
                          _ws(bse, plan, bse.BSE_WS_EPSM, nw))
    bse.bse_status_read(plan)
    eps = eps.cpu().numpy()
    for w in range(nw):
        c = chi[w].astype(np.complex128)
        M = np.eye(ng) - (c if F is None else c + c @ F.astype(np.complex128))
        x = np.linalg.solve(M, c[:, 0])
        dx = 8 * ng * 2.0 ** -24 * np.linalg.cond(M) * np.linalg.norm(x)
        # the kernel's product adds ng roundings of its entries
        if F is not None:
            dx += ng * 2.0 ** -24 * np.linalg.norm(np.linalg.inv(M), 2) * np.linalg.norm(np.abs(c) @ np.abs(F)) * np.linalg.norm(x)
        assert abs(1.0 / eps[w] - (1.0 + x[0])) <= dx, w


def test_screening_range_equals_single_points(bse):
    """W of a range (more q than one group of split images) is W of each q on its own, bit for bit."""
    spec = _spec(4, 1, 2, 2.0, 24)
    plan = bse.Plan([spec])
    inf = plan.info(0)
    nq, K, ng = inf["nq"], inf["dim"], inf["ng_max"]
    rng = np.random.default_rng(1)
    en = _dev(np.sort(rng.uniform(-0.3, 0.4, (inf["nkpt"], 3)), axis=1), torch.float64)
    P = _dev(rng.standard_normal(K) + 1j * rng.standard_normal(K), torch.complex128)
    rho = _dev(0.1 * (rng.standard_normal((nq * K, ng)) + 1j * rng.standard_normal((nq * K, ng))), torch.complex64)
    W, W1 = [torch.zeros(nq, ng, ng, dtype=torch.complex64, device="cuda") for _ in range(2)]
    res = torch.zeros(nq, device="cuda")
    bse.bse_screening(plan, 0, rho.clone(), en, P, 0, nq, 12, W, res, _ws(bse, plan, bse.BSE_WS_SCREEN, nq))
    for q in (0, 1, 31, 32, 33, nq - 1):
        one = rho[q * K:(q + 1) * K].clone()
        bse.bse_screening(plan, 0, one, en, P, q, q + 1, 12, W1, None, _ws(bse, plan, bse.BSE_WS_SCREEN, 1))
        bse.bse_status_read(plan)
        assert torch.equal(W1[q], W[q]), q
    assert float(res.max()) < 1e-4
    assert torch.equal(W, W.mH)
