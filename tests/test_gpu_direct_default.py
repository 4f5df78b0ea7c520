"""Route of the direct pair densities when no variant has been chosen: the tensor-core kernel where its tiles are
many and full enough, the correlation kernel elsewhere; both against the oracle's correlation in 64 bits.

Bound per entry of the tensor-core route, from the arithmetic (states are normalised, so the magnitudes of
the terms of an entry sum to at most 1): the split products are within 2^-21, each K chunk of 32 adds at most
12 truncations of 2^-23 of its own sum, and the promotion one rounding of 2^-24 per chunk.
"""
import numpy as np
import pytest

from oracle import pair as op
from synth import SystemSpec, generate

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


# (lattice, n, nv, nc, ecut, grid, q range, tensor route expected)
CELLS = [("fcc", 5, 4, 4, 3.0, (48, 48, 48), (0, 125), True),       # prime mesh: 5-point regions, ragged columns
         ("fcc", 6, 3, 4, 4.0, (32, 32, 32), (36, 144), True),      # whole planes of the mesh
         ("fcc", 6, 1, 2, 4.0, (32, 32, 32), (5, 209), True),       # a range that starts and ends inside a plane
         ("hex", 18, 1, 1, 2.5, (12, 12, 48), (0, 64), True),       # 54-point regions
         ("fcc", 6, 3, 4, 4.0, (32, 32, 32), (7, 9), False),        # two q: nearly empty tiles
         ("fcc", 3, 3, 2, 4.0, (24, 24, 24), (0, 27), False)]       # fewer tiles than SMs


@pytest.mark.parametrize("cell", CELLS, ids=lambda c: f"{c[0]}{c[1]}_{c[2]}v{c[3]}c_q{c[6][0]}-{c[6][1]}")
def test_default_route(bse, cell):
    lat, n, nv, nc, ecut, grid, (q0, q1), tensor = cell
    spec = SystemSpec("cell", lat, 10.0 if lat == "fcc" else 4.7, 30.0, (n, n, n if lat == "fcc" else 1), nv, nc, ecut,
                      grid, "3d" if lat == "fcc" else "slab", r0=20.0)
    s = generate(spec, with_w=False)
    plan = bse.Plan([spec])
    inf = plan.info(0)
    ws = torch.empty(bse.bse_workspace_size(plan, 0, bse.BSE_WS_PAIR) // 8 + 1, dtype=torch.complex64, device="cuda")
    coef = s.coef.astype(np.complex64)
    bse.bse_pair_densities(plan, 0, bse.BSE_PD_REALSPACE, _dev(coef, torch.complex64), None, None, None, None, 0, 0, ws)

    def densities(flags, variant):
        bse.bse_set_pair_variant(plan, 0, variant)
        out = torch.zeros(bse.bse_rho_dir_count(plan, 0, q0, q1), inf["ng_max"], dtype=torch.complex64, device="cuda")
        bse.bse_pair_densities(plan, 0, flags, None, None, None, None, out, q0, q1, ws)
        bse.bse_status_read(plan)
        return out.cpu().numpy()

    default = densities(bse.BSE_PD_DIRECT, -1)
    on_tensor = densities(bse.BSE_PD_DIRECT | bse.BSE_PD_TENSOR, -1)
    plain = densities(bse.BSE_PD_DIRECT, 64)
    assert np.array_equal(default, on_tensor if tensor else plain)
    tol = 2.0 ** -21 + 12 * 2.0 ** -23 + inf["tc_kpad"] // 32 * 2.0 ** -24
    rng = np.random.default_rng(5)
    at = 0
    for iq in range(q0, q1):
        blk, _ = bse.bse_pair_blocks(plan, 0, iq)
        ng, nb = len(bse.bse_gvectors(plan, 0, iq, True)), len(blk)
        for j in rng.choice(nb, min(2, nb), replace=False):
            _, rv, rc = op.direct_rho_block(spec, int(blk[j][0]), int(blk[j][1]), s.gk, coef.astype(np.complex128))
            v = on_tensor[at + j * nv * nv: at + (j + 1) * nv * nv, :ng].reshape(nv, nv, ng)
            c = on_tensor[at + nb * nv * nv + j * nc * nc: at + nb * nv * nv + (j + 1) * nc * nc, :ng].reshape(nc, nc, ng)
            assert max(np.abs(v - rv).max(), np.abs(c - rc).max()) <= tol, (iq, j)
        at += nb * (nv * nv + nc * nc)
