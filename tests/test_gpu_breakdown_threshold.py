"""The Haydock recursion's breakdown test b_{j+1} <= 1e-6 |H v_j| where |H v| jumps by a factor of 1000 from one step to
the next: a CTA that compared b with a partial sum of the next step would stop early (and leave the others waiting).

H = diag(1 on the first half, 1000 on the second) + delta (v0 w^H + w v0^H), v0 and w unit vectors of the two halves,
P = v0: b_1 = delta against |H v_0| = 1, while |H v_1| is about 1000.  The products see v_0 rounded to FP32, which adds a
residual of at most 2^-24 to b_1 (0.12 of the distance of delta from the threshold at most) and, as a part of v_1 outside the
span of v0 and w, keeps the recursion going past step 1.
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


@pytest.mark.parametrize("n,delta,stops", [(3, 2.0e-6, False), (6, 2.0e-6, False), (6, 5.0e-7, True)])
def test_threshold_uses_its_own_step(bse, n, delta, stops):
    spec = SystemSpec("cell", "fcc", 10.0, 0.0, (n, n, n), 2, 2, 1.0, (8, 8, 8), "3d")
    plan = bse.Plan([spec])
    dim = plan.info(0)["dim"]
    h = dim // 2
    rng = np.random.default_rng(7)
    z = rng.standard_normal((2, h)) + 1j * rng.standard_normal((2, h))
    z /= np.linalg.norm(z, axis=1, keepdims=True)
    H = np.zeros((dim, dim), dtype=np.complex128)
    H[np.arange(h), np.arange(h)] = 1.0
    H[np.arange(h, dim), np.arange(h, dim)] = 1000.0
    H[h:, :h] = delta * np.outer(z[1], z[0].conj())
    H[:h, h:] = H[h:, :h].conj().T
    P = np.zeros(dim, dtype=np.complex128)
    P[:h] = z[0]
    Hd = torch.as_tensor(H.astype(np.complex64), device="cuda")
    Pd = torch.as_tensor(P, device="cuda")
    nsteps = 6
    om = torch.linspace(0.0, 2.0, 16, dtype=torch.float64, device="cuda")
    ws = torch.empty(bse.bse_workspace_size(plan, 0, bse.BSE_WS_SPECTRUM, nsteps) // 8 + 1, dtype=torch.complex64,
                     device="cuda")
    first = None
    for _ in range(40):
        eps2 = torch.zeros(16, dtype=torch.float64, device="cuda")
        ab = torch.zeros(2 * nsteps, dtype=torch.float64, device="cuda")
        done = torch.zeros(1, dtype=torch.int32, device="cuda")
        bse.bse_spectrum(plan, 0, Hd, Pd, nsteps, om, 0.05, eps2, ab, done, ws)
        bse.bse_status_read(plan)
        assert (int(done.item()) == 1) == stops
        first = ab.clone() if first is None else first
        assert torch.equal(ab, first)
    if not stops:
        assert -2.0 ** -20 * delta <= float(first[nsteps + 1]) - delta <= 2.0 ** -24 + 2.0 ** -20 * delta
