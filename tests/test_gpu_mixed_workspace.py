"""The mixed build with a kernel workspace that starts 8 bytes past a 16-byte boundary (a complex64 slice): the same bits as
with an aligned one, at an odd and an even vector stride."""
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


@pytest.mark.parametrize("n,ecut", [(2, 4.0), (3, 4.0), (2, 2.5), (3, 1.6)])
def test_offset_workspace_same_bits(bse, n, ecut):
    spec = SystemSpec("cell", "fcc", 10.0, 0.0, (n, n, n), 3, 2, ecut, (24,) * 3, "3d")
    s = generate(spec, wdtype=np.complex64)
    plan = bse.Plan([spec])
    inf = plan.info(0)
    rng = np.random.default_rng(11)

    def rand(*shape):
        return torch.as_tensor((rng.standard_normal(shape) + 1j * rng.standard_normal(shape)).astype(np.complex64), device="cuda")
    rho_x, rho = rand(inf["dim"], inf["ng_max"]), rand(bse.bse_rho_dir_count(plan, 0, 0, inf["nq"]), inf["ng_max"])
    W = torch.as_tensor(s.W, dtype=torch.complex64, device="cuda")
    en = torch.as_tensor(s.energies, dtype=torch.float64, device="cuda")
    size = bse.bse_workspace_size(plan, 0, bse.BSE_WS_KERNEL, inf["nq"]) // 8 + 1
    out = []
    for off in (0, 1):
        ws = torch.empty(size + off, dtype=torch.complex64, device="cuda")[off:]
        assert ws.data_ptr() % 16 == 8 * off
        H = torch.zeros(inf["dim"], inf["dim"], dtype=torch.complex64, device="cuda")
        bse.bse_build_kernel(plan, 0, bse.BSE_BK_INIT | bse.BSE_BK_DIRECT, rho_x, rho, 0, inf["nq"], W, en, 0.1,
                             bse.BSE_PREC_BF16X3, H, ws)
        bse.bse_status_read(plan)
        out.append(H)
    assert bool(torch.isfinite(torch.view_as_real(out[0])).all()) and torch.equal(out[0], out[1])
