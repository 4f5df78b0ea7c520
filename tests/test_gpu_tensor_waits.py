"""Order of the tensor-core kernels' waits: a product issued, or an accumulator read, before the data it depends on is
visible changes single entries from run to run.  Builds whose rings and accumulators wrap many times, in both precisions,
repeated on a busy GPU: every run gives the same bits.
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


@pytest.mark.parametrize("n,nv,nc,ecut,grid", [(5, 4, 4, 3.0, 48), (6, 3, 4, 4.0, 32), (4, 4, 4, 13.0, 48)])
def test_repeated_builds_same_bits(bse, n, nv, nc, ecut, grid):
    from paper_1206_3518_gb300.pipeline import Forward
    spec = SystemSpec("cell", "fcc", 10.0, 0.0, (n, n, n), nv, nc, ecut, (grid,) * 3, "3d")
    s = generate(spec, wdtype=np.complex64)
    plan = bse.Plan([spec])
    F = Forward(plan, 0, nsteps=8, nw=8)
    coef = torch.as_tensor(s.coef, dtype=torch.complex64, device="cuda")
    en = torch.as_tensor(s.energies, dtype=torch.float64, device="cuda")
    W = torch.as_tensor(s.W, dtype=torch.complex64, device="cuda")
    for prec in (bse.BSE_PREC_FP32, bse.BSE_PREC_BF16X3):
        first = None
        for _ in range(12):
            F.H.fill_(float("nan"))
            F.build(coef, en, W, spec.delta, prec, tensor_pair=bool(plan.info(0)["tensor_pair"]))
            if first is None:
                first, rho = F.H.clone(), F.rho_dir.clone()
                assert bool(torch.isfinite(torch.view_as_real(first)).all())
            assert torch.equal(F.H, first) and torch.equal(F.rho_dir, rho)
        bse.bse_status_read(plan)
