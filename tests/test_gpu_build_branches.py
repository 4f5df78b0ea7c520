"""Branches of the FP32 build: the exchange term on the tensor cores (a workspace given) at dimensions around its
128-row tiles, the direct term's block products for every pair of band counts, and workspaces that start eight
bytes off a 16-byte boundary.

Bounds per entry, from the arithmetic, relative to the sum of the magnitudes of the terms.  Exchange: rounding of
the scaled densities 2 x 2^-24, split products 2^-21, per chunk of 32 complex K at most 12 truncations of 2^-23 and the
promotion 2^-24, plus one rounding for the diagonal.  Block product: 2 NG roundings of 2^-24 on top of W.rho's bound
(split 2^-21, 12 truncations, a promotion per chunk).
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


def _cplx(rng, *shape):
    return rng.standard_normal(shape) + 1j * rng.standard_normal(shape)


def _ws(bse, plan, kind, arg=0, off=0):
    n = bse.bse_workspace_size(plan, 0, kind, arg) // 8 + 1
    return torch.empty(n + off, dtype=torch.complex64, device="cuda")[off:]


def _fcc(n, nv, nc, ecut, grid):
    return SystemSpec("cell", "fcc", 10.0, 0.0, (n, n, n), nv, nc, ecut, (grid,) * 3, "3d")


# dimensions 8, 72, 128, 243, 216 and 256
@pytest.mark.parametrize("n,nv,nc,ecut,grid", [(2, 1, 1, 1.0, 8), (2, 3, 3, 1.6, 24), (2, 4, 4, 4.0, 24), (3, 3, 3, 1.0, 8),
                                               (3, 2, 4, 4.0, 24), (4, 2, 2, 8.6, 32)])
def test_exchange_term_with_a_workspace(bse, n, nv, nc, ecut, grid):
    plan = bse.Plan([_fcc(n, nv, nc, ecut, grid)])
    inf = plan.info(0)
    dim, ngm, nk, nvc = inf["dim"], inf["ng_max"], n ** 3, nv * nc
    rng = np.random.default_rng(5)
    rho = (_cplx(rng, dim, ngm) * 10.0 ** rng.uniform(-3, 3, (dim, 1))).astype(np.complex64)
    rho[dim // 2] = 0.0
    e = np.sort(rng.uniform(-1, 1, (nk, nv + nc)), axis=1)
    dev = "cuda"
    r, en = torch.as_tensor(rho, device=dev), torch.as_tensor(e, device=dev)
    out = []
    for ws in (None, _ws(bse, plan, bse.BSE_WS_KERNEL, 1), _ws(bse, plan, bse.BSE_WS_KERNEL, 1, off=1)):
        H = torch.zeros(dim, dim, dtype=torch.complex64, device=dev)
        bse.bse_build_kernel(plan, 0, bse.BSE_BK_INIT | bse.BSE_BK_MIRROR, r, None, 0, 0, None, en, 0.1, bse.BSE_PREC_FP32,
                             H, ws)
        bse.bse_status_read(plan)
        out.append(H.cpu().numpy())
    assert np.array_equal(out[1], out[2])
    g = bse.bse_gvectors(plan, 0, 0, True)
    ng = len(g)
    # the scale of the exchange term from the kernel without a workspace: H of one unit entry per G
    x = rho[:, :ng].astype(np.complex128)
    s2 = np.zeros(ng)
    unit = torch.zeros(dim, ngm, dtype=torch.complex64, device=dev)
    for j in range(ng):
        unit.zero_()
        unit[0, j] = unit[1 if dim > 1 else 0, j] = 1.0
        H = torch.zeros(dim, dim, dtype=torch.complex64, device=dev)
        bse.bse_build_kernel(plan, 0, bse.BSE_BK_INIT, unit, None, 0, 0, None, en, 0.1, bse.BSE_PREC_FP32, H, None)
        s2[j] = H[0, 1].real.item()
    ref = (x.conj() * s2) @ x.T
    size = 2.0 * ((np.abs(x) * s2) @ np.abs(x).T)
    k = np.arange(dim) // nvc
    de = (e[:, None, nv:] - e[:, :nv, None]).reshape(-1) + 0.1
    ref[np.arange(dim), np.arange(dim)] += de
    size[np.arange(dim), np.arange(dim)] += np.abs(de)
    tol = 2.0 ** -21 + 12 * 2.0 ** -23 + (ng / 32 + 8) * 2.0 ** -24
    up = k[:, None] <= k[None, :]
    assert np.all(np.abs(out[1] - ref)[up] <= (tol * size)[up] + 1e-30)
    assert np.allclose(out[1], out[1].conj().T, rtol=0, atol=0)


@pytest.mark.parametrize("nv", [1, 2, 3, 4])
@pytest.mark.parametrize("nc", [1, 2, 3, 4])
@pytest.mark.parametrize("off", [0, 1])
def test_block_products_of_all_band_counts(bse, nv, nc, off):
    plan = bse.Plan([_fcc(2, nv, nc, 1.6, 24)])
    inf = plan.info(0)
    nq, ngm, dim, nvc = inf["nq"], inf["ng_max"], inf["dim"], nv * nc
    rng = np.random.default_rng(17)
    rho = _cplx(rng, bse.bse_rho_dir_count(plan, 0, 0, nq), ngm).astype(np.complex64)
    W = _cplx(rng, nq, ngm, ngm)
    W = (W + W.conj().transpose(0, 2, 1)).astype(np.complex64)
    H = torch.zeros(dim, dim, dtype=torch.complex64, device="cuda")
    bse.bse_build_kernel(plan, 0, bse.BSE_BK_DIRECT, None, torch.as_tensor(rho, device="cuda"), 0, nq,
                         torch.as_tensor(W, device="cuda"), None, 0.0, bse.BSE_PREC_FP32, H,
                         _ws(bse, plan, bse.BSE_WS_KERNEL, nq, off))
    bse.bse_status_read(plan)
    H, at = H.cpu().numpy(), 0
    for iq in range(nq):
        blk, _ = bse.bse_pair_blocks(plan, 0, iq)
        ng, nb = len(bse.bse_gvectors(plan, 0, iq, True)), len(blk)
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
            assert np.array_equal(H[k2 * nvc:(k2 + 1) * nvc, k * nvc:(k + 1) * nvc], got.conj().T) or k == k2
