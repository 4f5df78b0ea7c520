"""H of the FP32 build does not depend on how the q mesh is cut, also on meshes whose direct densities take the tensor cores:
chunks of a build give the single pass's bits, and so do the densities of a split's per-q calls."""
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


@pytest.mark.parametrize("lat,n,nv,nc,ecut,grid,chunks", [("fcc", 5, 4, 4, 3.0, (48,) * 3, (7, 25, 100)),
                                                          ("hex", 18, 1, 2, 2.5, (12, 12, 48), (1, 64)),
                                                          ("fcc", 4, 3, 3, 4.0, (24,) * 3, (5,))])
def test_chunked_builds_equal_the_single_pass(bse, lat, n, nv, nc, ecut, grid, chunks):
    from paper_1206_3518_gb300 import shard
    from paper_1206_3518_gb300.pipeline import Forward
    spec = SystemSpec("cell", lat, 10.0 if lat == "fcc" else 4.7, 30.0, (n, n, n if lat == "fcc" else 1), nv, nc, ecut,
                      grid, "3d" if lat == "fcc" else "slab", r0=20.0)
    s = generate(spec, wdtype=np.complex64)
    plan = bse.Plan([spec])
    coef = torch.as_tensor(s.coef, dtype=torch.complex64, device="cuda")
    en = torch.as_tensor(s.energies, dtype=torch.float64, device="cuda")
    W = torch.as_tensor(s.W, dtype=torch.complex64, device="cuda")
    F = Forward(plan, 0, nsteps=8, nw=8)
    ref = F.build(coef, en, W, spec.delta).clone()
    nq = plan.info(0)["nq"]
    for c in chunks:
        assert torch.equal(Forward(plan, 0, nsteps=8, nw=8, qchunk=c).build(coef, en, W, spec.delta), ref), c
    # the ranks of a split: one q at a time, the densities of the single pass
    bse.bse_pair_densities(plan, 0, shard.direct_flags(plan), None, None, None, None, F.rho_dir, 0, nq, F.ws_pair)
    for q in range(0, nq, max(1, nq // 17)):
        a, n1 = bse.bse_rho_dir_count(plan, 0, 0, q) if q else 0, bse.bse_rho_dir_count(plan, 0, q, q + 1)
        out = torch.zeros(n1, F.ng_max, dtype=torch.complex64, device="cuda")
        bse.bse_pair_densities(plan, 0, shard.direct_flags(plan), None, None, None, None, out, q, q + 1, F.ws_pair)
        ng = len(bse.bse_gvectors(plan, 0, q, 1))
        assert torch.equal(out[:, :ng], F.rho_dir[a:a + n1, :ng]), q
    bse.bse_status_read(plan)


def test_no_tensor_cores_asked_for(bse):
    """tensor_pair=False takes the variant in use in every chunk, also where the tensor cores are the default."""
    from paper_1206_3518_gb300.pipeline import Forward
    spec = SystemSpec("cell", "fcc", 10.0, 0.0, (5, 5, 5), 4, 4, 3.0, (48,) * 3, "3d")
    s = generate(spec, wdtype=np.complex64)
    plan = bse.Plan([spec])
    assert bse.bse_pair_route(plan, 0, 0, 125)
    args = (torch.as_tensor(s.coef, dtype=torch.complex64, device="cuda"),
            torch.as_tensor(s.energies, dtype=torch.float64, device="cuda"),
            torch.as_tensor(s.W, dtype=torch.complex64, device="cuda"), spec.delta)
    for prec in (bse.BSE_PREC_FP32, bse.BSE_PREC_BF16X3):
        F = Forward(plan, 0, nsteps=8, nw=8)
        H = F.build(*args, prec, tensor_pair=False).clone()
        rho = F.rho_dir.clone()
        bse.bse_set_pair_variant(plan, 0, 64)
        bse.bse_pair_densities(plan, 0, bse.BSE_PD_DIRECT, None, None, None, None, F.rho_dir, 0, 125, F.ws_pair)
        assert torch.equal(F.rho_dir, rho)
        bse.bse_set_pair_variant(plan, 0, -1)
        assert torch.equal(Forward(plan, 0, nsteps=8, nw=8, qchunk=30).build(*args, prec, tensor_pair=False), H)
    with pytest.raises(bse.BseError):
        bse.bse_pair_densities(plan, 0, bse.BSE_PD_DIRECT | bse.BSE_PD_TENSOR | bse.BSE_PD_VARIANT, None, None, None, None,
                               F.rho_dir, 0, 125, F.ws_pair)
    bse.bse_status_read(plan)
