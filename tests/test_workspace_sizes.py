"""Workspaces whose products keep split images of their operands: the images are bounded whatever the system (host plans)."""
import pytest

from synth import SystemSpec

from paper_1206_3518_gb300 import bse

GIB = 1 << 30


def _plan(n, nv, nc, ecut, grid):
    return bse.Plan([SystemSpec("cell", "fcc", 10.0, 0.0, (n, n, n), nv, nc, ecut, (grid,) * 3, "3d")], host_only=True)


def _a256(x):
    return (x + 255) // 256 * 256


@pytest.mark.parametrize("nw", [1, 7, 2000])
def test_dyson_holds_the_systems_and_one_vector_each(nw):
    plan = _plan(2, 3, 4, 8.6, 32)
    n = plan.info(0)["ng0"]
    assert bse.bse_workspace_size(plan, 0, bse.BSE_WS_EPSM, nw) == _a256(nw * n * (n + 1) * 8) + _a256(nw * n * 8)


@pytest.mark.parametrize("n,nv,nc,ecut,grid", [(2, 1, 1, 12.0, 48), (2, 4, 4, 12.0, 48), (6, 3, 4, 8.6, 32)])
def test_chi0_images_and_sums(n, nv, nc, ecut, grid):
    plan = _plan(n, nv, nc, ecut, grid)
    inf = plan.info(0)
    vectors = inf["ng0"] * (inf["dim"] + 64) * 8 + inf["dim"] * 8
    weights = 4 * 1024 * 4 * (inf["dim"] + 64)
    size = bse.bse_workspace_size(plan, 0, bse.BSE_WS_CHI0)
    assert size <= vectors + weights + GIB // 2 + (1 << 22)


@pytest.mark.parametrize("n,nv,nc,ecut,grid", [(4, 4, 4, 12.0, 48), (8, 4, 4, 8.6, 48), (8, 3, 4, 8.6, 32)])
def test_backward_images(n, nv, nc, ecut, grid):
    plan = _plan(n, nv, nc, ecut, grid)
    inf = plan.info(0)
    dim, ng, nk, ns, nq = inf["dim"], inf["ng_max"], inf["nkpt"], 300, min(32, inf["nq"])
    rows = min(nq * nk, inf["nblocks"])
    own = (bse.bse_workspace_size(plan, 0, bse.BSE_WS_SPECTRUM, ns) + 8 * dim * dim + 16 * ns * dim + 16 * ns * ns
           + 8 * rows * (nv * nv + 2 * nc * nc) * ng)
    panel = 8 * (min(dim, 4096) + 128) * (dim + 32) + 8 * (inf["ng0"] + 128) * (dim + 32)
    assert bse.bse_workspace_size(plan, 0, bse.BSE_WS_BACKWARD, ns) <= own + max(3 * GIB // 2 + (1 << 24), panel) + (1 << 25)
