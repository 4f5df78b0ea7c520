"""The split products over FP32's whole range: rows near its largest numbers times rows near its smallest, whose products are
ordinary numbers.  Bounds as in the tests of the products at ordinary sizes: split products 2^-21, a chunk of K adds at most
24 truncations of 2^-23, promotion and block product one rounding of 2^-24 per term, relative to the terms' magnitudes.
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
    return rng.uniform(-1, 1, shape) + 1j * rng.uniform(-1, 1, shape)


# powers of two of the rows that W multiplies, of W and of the other rows
@pytest.mark.parametrize("pr,pw,po", [(126, -120, 0), (127, -126, 0), (110, -20, -90), (-105, 110, 0), (-120, 100, 20),
                                      (58, 58, -100), (-60, -60, 110)])
@pytest.mark.parametrize("nv,nc", [(1, 2), (2, 1)])
def test_direct_term(bse, nv, nc, pr, pw, po):
    plan = bse.Plan([SystemSpec("cell", "fcc", 10.0, 0.0, (2, 2, 2), nv, nc, 1.6, (24,) * 3, "3d")])
    inf = plan.info(0)
    nq, ngm, dim, nvc = inf["nq"], inf["ng_max"], inf["dim"], nv * nc
    rng = np.random.default_rng(23)
    nvec = bse.bse_rho_dir_count(plan, 0, 0, nq)
    rho, at = _cplx(rng, nvec, ngm), 0
    spans = []
    for iq in range(nq):
        nb = len(bse.bse_pair_blocks(plan, 0, iq)[0])
        spans.append((at, nb))
        v, c = slice(at, at + nb * nv * nv), slice(at + nb * nv * nv, at + nb * (nv * nv + nc * nc))
        rho[v] *= 2.0 ** (pr if nv < nc else po)
        rho[c] *= 2.0 ** (po if nv < nc else pr)
        at = c.stop
    rho = rho.astype(np.complex64)
    W = _cplx(rng, nq, ngm, ngm)
    W = ((W + W.conj().transpose(0, 2, 1)) * 2.0 ** (pw - 1)).astype(np.complex64)
    assert np.isfinite(rho).all() and np.isfinite(W).all()
    H = torch.zeros(dim, dim, dtype=torch.complex64, device="cuda")
    ws = torch.empty(bse.bse_workspace_size(plan, 0, bse.BSE_WS_KERNEL, nq) // 8 + 1, dtype=torch.complex64, device="cuda")
    bse.bse_build_kernel(plan, 0, bse.BSE_BK_DIRECT, None, torch.as_tensor(rho, device="cuda"), 0, nq,
                         torch.as_tensor(W, device="cuda"), None, 0.0, bse.BSE_PREC_FP32, H, ws)
    bse.bse_status_read(plan)
    H = H.cpu().numpy()
    for iq, (at, nb) in enumerate(spans):
        blk, _ = bse.bse_pair_blocks(plan, 0, iq)
        ng = len(bse.bse_gvectors(plan, 0, iq, True))
        rv = rho[at: at + nb * nv * nv, :ng].astype(np.complex128).reshape(nb, nv * nv, ng)
        rc = rho[at + nb * nv * nv: at + nb * (nv * nv + nc * nc), :ng].astype(np.complex128).reshape(nb, nc * nc, ng)
        w = W[iq, :ng, :ng].astype(np.complex128)
        tol = 2.0 ** -21 + 24 * 2.0 ** -23 + (4 * ng + ng / 32) * 2.0 ** -24
        for b, (k, k2) in enumerate(blk):
            m = -inf["norm"] * (rv[b].conj() @ w @ rc[b].T)
            size = 2.0 * inf["norm"] * (np.abs(rv[b]) @ np.abs(w) @ np.abs(rc[b]).T)
            m, size = [x.reshape(nv, nv, nc, nc).transpose(0, 2, 1, 3).reshape(nvc, nvc) for x in (m, size)]
            if k == k2:
                m, size = 0.5 * (m + m.conj().T), 0.5 * (size + size.T)
            got = H[k * nvc:(k + 1) * nvc, k2 * nvc:(k2 + 1) * nvc]
            assert np.all(np.abs(got - m) <= tol * size), (iq, b)


@pytest.mark.parametrize("big,small", [(126, -126), (100, -90), (64, -40)])
def test_pair_densities(bse, big, small):
    from oracle import pair as op
    n, nv, nc = 3, 2, 2
    spec = SystemSpec("cell", "fcc", 10.0, 0.0, (n, n, n), nv, nc, 2.5, (24,) * 3, "3d")
    plan = bse.Plan([spec])
    inf = plan.info(0)
    nq, nk = inf["nq"], inf["nkpt"]
    assert inf["tensor_pair"] == 1
    rng = np.random.default_rng(29)
    gk = [bse.bse_gvectors(plan, 0, k, 0) for k in range(nk)]
    c = np.zeros((nk, nv + nc, inf["npw_max"]), dtype=np.complex128)
    for k in range(nk):
        c[k, :, : len(gk[k])] = _cplx(rng, nv + nc, len(gk[k])) / np.sqrt(len(gk[k]))
    c[:, 0::2] *= 2.0 ** big                             # bands 0 and 2 large, 1 and 3 small
    c[:, 1::2] *= 2.0 ** small
    c = c.astype(np.complex64)
    ws = torch.empty(bse.bse_workspace_size(plan, 0, bse.BSE_WS_PAIR) // 8 + 1, dtype=torch.complex64, device="cuda")
    bse.bse_pair_densities(plan, 0, bse.BSE_PD_REALSPACE, torch.as_tensor(c, device="cuda"), None, None, None, None, 0, 0, ws)
    out = torch.zeros(bse.bse_rho_dir_count(plan, 0, 0, nq), inf["ng_max"], dtype=torch.complex64, device="cuda")
    bse.bse_pair_densities(plan, 0, bse.BSE_PD_DIRECT | bse.BSE_PD_TENSOR, None, None, None, None, out, 0, nq, ws)
    bse.bse_status_read(plan)
    out, at = out.cpu().numpy(), 0
    tol = (2.0 ** -21 + 24 * 2.0 ** -23 + inf["tc_kpad"] / 32 * 2.0 ** -24) * 2.0 ** (big + small) * 2.0
    for iq in range(nq):
        blk, _ = bse.bse_pair_blocks(plan, 0, iq)
        ng, nb = len(bse.bse_gvectors(plan, 0, iq, True)), len(blk)
        for j in range(0, nb, 5):
            _, rv, rc = op.direct_rho_block(spec, int(blk[j][0]), int(blk[j][1]), gk, c.astype(np.complex128))
            v = out[at + j * nv * nv: at + (j + 1) * nv * nv, :ng].reshape(nv, nv, ng)
            w = out[at + nb * nv * nv + j * nc * nc: at + nb * nv * nv + (j + 1) * nc * nc, :ng].reshape(nc, nc, ng)
            for a, b in ((0, 1), (1, 0)):                # large times small
                assert max(np.abs(v[a, b] - rv[a, b]).max(), np.abs(w[a, b] - rc[a, b]).max()) <= tol, (iq, j)
        at += nb * (nv * nv + nc * nc)


@pytest.mark.parametrize("big", [10, 18, 24])
def test_large_component_meets_zeros(bse, big):
    """Rows of rho and W whose largest component (G = 0, 2^big above the rest) meets zeros of the other operand, as the head of
    W and the overlaps do where the wings vanish.  A component a of a row with largest m is kept to 2^-22 |a| + 2^-40 m."""
    nv, nc = 2, 3
    plan = bse.Plan([SystemSpec("cell", "fcc", 10.0, 0.0, (2, 2, 2), nv, nc, 2.5, (24,) * 3, "3d")])
    inf = plan.info(0)
    nq, ngm, dim, nvc = inf["nq"], inf["ng_max"], inf["dim"], nv * nc
    rng = np.random.default_rng(31)
    rho = _cplx(rng, bse.bse_rho_dir_count(plan, 0, 0, nq), ngm)
    rho[:, 0] *= 2.0 ** big
    rho = rho.astype(np.complex64)
    W = _cplx(rng, nq, ngm, ngm)
    W = W + W.conj().transpose(0, 2, 1)
    W[:, 0, :] = 0.0
    W[:, :, 0] = 0.0                                     # the head too: nothing of the large component is left
    W = W.astype(np.complex64)
    H = torch.zeros(dim, dim, dtype=torch.complex64, device="cuda")
    ws = torch.empty(bse.bse_workspace_size(plan, 0, bse.BSE_WS_KERNEL, nq) // 8 + 1, dtype=torch.complex64, device="cuda")
    bse.bse_build_kernel(plan, 0, bse.BSE_BK_DIRECT, None, torch.as_tensor(rho, device="cuda"), 0, nq,
                         torch.as_tensor(W, device="cuda"), None, 0.0, bse.BSE_PREC_FP32, H, ws)
    bse.bse_status_read(plan)
    H, at = H.cpu().numpy(), 0
    for iq in range(nq):
        blk, _ = bse.bse_pair_blocks(plan, 0, iq)
        ng, nb = len(bse.bse_gvectors(plan, 0, iq, True)), len(blk)
        rv = rho[at: at + nb * nv * nv, :ng].astype(np.complex128).reshape(nb, nv * nv, ng)
        rc = rho[at + nb * nv * nv: at + nb * (nv * nv + nc * nc), :ng].astype(np.complex128).reshape(nb, nc * nc, ng)
        at += nb * (nv * nv + nc * nc)
        w = W[iq, :ng, :ng].astype(np.complex128)
        tol = 2.0 ** -21 + 24 * 2.0 ** -23 + (4 * ng + ng / 32) * 2.0 ** -24
        for b, (k, k2) in enumerate(blk):
            m = -inf["norm"] * (rv[b].conj() @ w @ rc[b].T)
            kept = np.abs(rv[b]) * tol + 2.0 ** -39 * np.abs(rv[b]).max(axis=1, keepdims=True)     # W multiplies rho_vv'
            kept[:, 0] = 0.0                             # meets zeros only
            err = 2.0 * inf["norm"] * (kept @ np.abs(w) @ np.abs(rc[b]).T)
            m, err = [x.reshape(nv, nv, nc, nc).transpose(0, 2, 1, 3).reshape(nvc, nvc) for x in (m, err)]
            if k == k2:
                m, err = 0.5 * (m + m.conj().T), 0.5 * (err + err.T)
            got = H[k * nvc:(k + 1) * nvc, k2 * nvc:(k2 + 1) * nvc]
            assert np.all(np.abs(got - m) <= err), (iq, b)
