"""The default route of the direct densities (host tables only): where a part of the mesh takes the tensor cores the whole does,
so one flag per build says it; chosen variants and bad ranges."""
import pytest

from synth import SystemSpec

from paper_1206_3518_gb300 import bse, shard


def _plan(lat, n, nv, nc, ecut, grid):
    return bse.Plan([SystemSpec("cell", lat, 10.0 if lat == "fcc" else 4.7, 30.0, (n, n, n if lat == "fcc" else 1), nv, nc,
                                ecut, grid, "3d" if lat == "fcc" else "slab", r0=20.0)], host_only=True)


@pytest.mark.parametrize("lat,n,nv,nc,ecut,grid", [("fcc", 3, 3, 2, 4.0, (24,) * 3), ("fcc", 4, 3, 3, 4.0, (24,) * 3),
                                                   ("fcc", 5, 4, 4, 3.0, (48,) * 3), ("fcc", 6, 1, 2, 4.0, (32,) * 3),
                                                   ("fcc", 7, 2, 2, 3.0, (24,) * 3), ("hex", 18, 1, 1, 2.5, (12, 12, 48)),
                                                   ("hex", 19, 1, 3, 2.5, (12, 12, 48)), ("hex", 24, 2, 2, 2.5, (12, 12, 48))])
def test_a_part_on_the_tensor_cores_means_the_whole(lat, n, nv, nc, ecut, grid):
    plan = _plan(lat, n, nv, nc, ecut, grid)
    nq = plan.info(0)["nq"]
    whole = bse.bse_pair_route(plan, 0, 0, nq)
    for step in (1, 2, 3, 7, 16, n, 2 * n, n * n):
        for a in range(0, nq - step + 1, max(1, step // 2)):
            assert whole or not bse.bse_pair_route(plan, 0, a, a + step)
    flags = shard.direct_flags(plan)
    assert flags == (bse.BSE_PD_DIRECT | (bse.BSE_PD_TENSOR if whole else bse.BSE_PD_VARIANT))
    bse.bse_set_pair_variant(plan, 0, 64)
    assert not bse.bse_pair_route(plan, 0, 0, nq)
    bse.bse_set_pair_variant(plan, 0, -1)
    for a, b in ((-1, 1), (0, nq + 1), (3, 3)):
        with pytest.raises(bse.BseError):
            bse.bse_pair_route(plan, 0, a, b)


def test_chosen_variant_and_the_tensor_form():
    plan = _plan("fcc", 5, 4, 4, 3.0, (48,) * 3)
    nq = plan.info(0)["nq"]
    assert bse.bse_pair_route(plan, 0, 0, nq)
    bse.bse_set_pair_variant(plan, 0, 64)
    assert not bse.bse_pair_route(plan, 0, 0, nq)
    bse.bse_set_pair_tensor(plan, 0, True)
    assert bse.bse_pair_route(plan, 0, 0, nq) and bse.bse_pair_variants(plan, 0)[1] == 64
    bse.bse_set_pair_variant(plan, 0, -1)
    assert bse.bse_pair_route(plan, 0, 0, nq)
