"""FP32 W.rho products on the tensor cores (FP16x3, promoted accumulation) against 64-bit products.

The direct term alone (BSE_BK_DIRECT on a zero H) of random pair densities and W, at sphere sizes on both
sides of the K16 step, the K chunk of 32, one N tile and several, with rows of very different size and a
zero row.  Bound per entry, from the arithmetic: every product of the split operands is within 2^-21 of its
size, a chunk of K adds at most 12 truncations of 2^-23 and the promotion and the block product one
rounding of 2^-24 per term, all relative to the sum of the magnitudes of the terms.
"""
import numpy as np
import pytest

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


# (lattice, n, nv, nc, ecut, grid): spheres of 15 to 530 points
CELLS = [("fcc", 2, 1, 2, 1.0, (8, 8, 8)), ("fcc", 2, 2, 1, 1.6, (24, 24, 24)), ("fcc", 3, 3, 2, 4.0, (24, 24, 24)),
         ("hex", 5, 2, 3, 2.5, (12, 12, 48)), ("fcc", 2, 3, 4, 8.6, (32, 32, 32)), ("fcc", 2, 4, 4, 12.0, (48, 48, 48))]


@pytest.mark.parametrize("cell", CELLS, ids=lambda c: f"{c[0]}{c[1]}_{c[2]}v{c[3]}c_{c[4]}Ha")
def test_direct_term_of_random_densities(bse, cell):
    from synth import SystemSpec
    lat, n, nv, nc, ecut, grid = cell
    spec = SystemSpec("cell", lat, 10.0 if lat == "fcc" else 4.7, 30.0, (n, n, n if lat == "fcc" else 1), nv, nc, ecut,
                      grid, "3d" if lat == "fcc" else "slab")
    plan = bse.Plan([spec])
    inf = plan.info(0)
    nq, ng_max, dim = inf["nq"], inf["ng_max"], inf["dim"]
    rng = np.random.default_rng(11)

    def cplx(*shape):
        return rng.standard_normal(shape) + 1j * rng.standard_normal(shape)

    nvec = bse.bse_rho_dir_count(plan, 0, 0, nq)
    rho = (cplx(nvec, ng_max) * 10.0 ** rng.uniform(-4, 4, (nvec, 1))).astype(np.complex64)
    rho[min(3, nvec - 1)] = 0.0
    W = cplx(nq, ng_max, ng_max) * 10.0 ** rng.uniform(-2, 2, (nq, ng_max, 1))
    W = (W + W.conj().transpose(0, 2, 1)).astype(np.complex64)
    dev = "cuda"
    H = torch.zeros(dim, dim, dtype=torch.complex64, device=dev)
    ws = torch.empty(bse.bse_workspace_size(plan, 0, bse.BSE_WS_KERNEL, nq) // 8 + 1, dtype=torch.complex64, device=dev)
    bse.bse_build_kernel(plan, 0, bse.BSE_BK_DIRECT, None, torch.as_tensor(rho, device=dev), 0, nq,
                         torch.as_tensor(W, device=dev), None, 0.0, bse.BSE_PREC_FP32, H, ws)
    bse.bse_status_read(plan)
    H = H.cpu().numpy()
    at, nvc = 0, nv * nc
    for iq in range(nq):
        blk, _ = bse.bse_pair_blocks(plan, 0, iq)
        ng = len(bse.bse_gvectors(plan, 0, iq, True))
        nb = len(blk)
        rv = rho[at: at + nb * nv * nv, :ng].astype(np.complex128).reshape(nb, nv * nv, ng)
        rc = rho[at + nb * nv * nv: at + nb * (nv * nv + nc * nc), :ng].astype(np.complex128).reshape(nb, nc * nc, ng)
        at += nb * (nv * nv + nc * nc)
        w = W[iq, :ng, :ng].astype(np.complex128)
        tol = 2.0 ** -21 + 12 * 2.0 ** -23 + (4 * ng + ng / 32) * 2.0 ** -24
        for b, (k, k2) in enumerate(blk):
            m = -inf["norm"] * (rv[b].conj() @ w @ rc[b].T)
            size = 2.0 * inf["norm"] * (np.abs(rv[b]) @ np.abs(w) @ np.abs(rc[b]).T)
            m, size = [x.reshape(nv, nv, nc, nc).transpose(0, 2, 1, 3).reshape(nvc, nvc) for x in (m, size)]
            if k == k2:
                m, size = 0.5 * (m + m.conj().T), 0.5 * (size + size.T)
            got = H[k * nvc:(k + 1) * nvc, k2 * nvc:(k2 + 1) * nvc]
            assert np.all(np.abs(got - m) <= tol * size + 1e-30), (iq, b)
            mirror = H[k2 * nvc:(k2 + 1) * nvc, k * nvc:(k + 1) * nvc]
            assert np.array_equal(mirror, got.conj().T) or k == k2
