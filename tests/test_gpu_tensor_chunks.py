"""Direct pair densities on the tensor cores against the correlation kernel at K layouts that end anywhere in a stage of
64 complex K, with boxes large enough that a stage holds one panel, over q ranges that leave most tiles empty.

Bound per entry, from the arithmetic (states are normalised, so the magnitudes of the terms of an entry sum to at
most 1): the split products are within 2^-21, each K chunk adds at most 24 truncations of 2^-23 of its own sum and
a rounding of 2^-24 on promotion; the correlation kernel's chains round four times per term, 2^-24 each.
"""
import numpy as np
import pytest

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


@pytest.mark.parametrize("n,nv,nc,ecut,grid", [(3, 2, 3, 1.0, 24), (4, 2, 3, 1.6, 24), (4, 1, 2, 2.5, 24), (4, 3, 3, 4.0, 24),
                                               (5, 2, 2, 6.0, 32), (4, 3, 4, 8.6, 32), (4, 4, 4, 13.0, 48), (4, 4, 4, 14.0, 48),
                                               (4, 4, 4, 15.0, 48)])
def test_chunks_and_empty_tiles(bse, n, nv, nc, ecut, grid):
    spec = SystemSpec("cell", "fcc", 10.0, 0.0, (n, n, n), nv, nc, ecut, (grid,) * 3, "3d")
    s = generate(spec, with_w=False)
    plan = bse.Plan([spec])
    inf = plan.info(0)
    if not inf["tensor_pair"]:
        pytest.skip("the tensor-core route is not built for this system")
    nq = inf["nq"]
    ws = torch.empty(bse.bse_workspace_size(plan, 0, bse.BSE_WS_PAIR) // 8 + 1, dtype=torch.complex64, device="cuda")
    coef = torch.as_tensor(np.ascontiguousarray(s.coef.astype(np.complex64)), device="cuda")
    bse.bse_pair_densities(plan, 0, bse.BSE_PD_REALSPACE, coef, None, None, None, None, 0, 0, ws)
    tol = 2.0 ** -21 + 24 * 2.0 ** -23 + (inf["tc_kpad"] / 32 + 4 * inf["tc_kpad"]) * 2.0 ** -24
    for q0, q1 in ((0, nq), (nq // 2, nq // 2 + 1), (nq - 2, nq)):
        out = []
        for flags, variant in ((bse.BSE_PD_DIRECT | bse.BSE_PD_TENSOR, -1), (bse.BSE_PD_DIRECT, 64)):
            bse.bse_set_pair_variant(plan, 0, variant)
            rho = torch.zeros(bse.bse_rho_dir_count(plan, 0, q0, q1), inf["ng_max"], dtype=torch.complex64, device="cuda")
            bse.bse_pair_densities(plan, 0, flags, None, None, None, None, rho, q0, q1, ws)
            bse.bse_status_read(plan)
            out.append(rho)
        assert float((out[0] - out[1]).abs().max()) <= tol, (q0, q1)
        assert float(out[0].abs().max()) > 0.0
