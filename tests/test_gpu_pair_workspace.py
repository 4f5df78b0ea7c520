"""The stages after BSE_PD_REALSPACE only read the pair workspace: calls for different q ranges that share one may overlap, and
the tiles of a range are dealt from the plan's tables alone, also where a range takes several launches.

Bound of the comparison with the correlation kernel, from the arithmetic (coefficient rows of norm 1, so the magnitudes
of the terms of an entry sum to at most 1): split products 2^-21, each K chunk 24 truncations of 2^-23 of its own sum
and a rounding of 2^-24 on promotion; the correlation kernel's chains round four times per term, 2^-24 each.
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


def _prepare(bse, lat, n, nv, nc, ecut, grid):
    spec = SystemSpec("cell", lat, 10.0 if lat == "fcc" else 4.7, 30.0, (n, n, n if lat == "fcc" else 1), nv, nc, ecut,
                      grid, "3d" if lat == "fcc" else "slab", r0=20.0)
    plan = bse.Plan([spec])
    inf = plan.info(0)
    assert inf["tensor_pair"] == 1
    gen = torch.Generator(device="cuda").manual_seed(9)
    c = torch.view_as_complex(torch.randn(inf["nkpt"], nv + nc, inf["npw_max"], 2, generator=gen, device="cuda"))
    npw = torch.as_tensor([len(bse.bse_gvectors(plan, 0, k, 0)) for k in range(inf["nkpt"])], device="cuda")
    c *= torch.arange(inf["npw_max"], device="cuda")[None, None, :] < npw[:, None, None]
    c /= torch.linalg.vector_norm(c, dim=2, keepdim=True)
    ws = torch.empty(bse.bse_workspace_size(plan, 0, bse.BSE_WS_PAIR) // 8 + 1, dtype=torch.complex64, device="cuda")
    bse.bse_pair_densities(plan, 0, bse.BSE_PD_REALSPACE, c.contiguous(), None, None, None, None, 0, 0, ws)
    return plan, inf, ws


def _direct(bse, plan, inf, ws, q0, q1, flags, out=None):
    if out is None:
        out = torch.zeros(bse.bse_rho_dir_count(plan, 0, q0, q1), inf["ng_max"], dtype=torch.complex64, device="cuda")
    bse.bse_pair_densities(plan, 0, flags, None, None, None, None, out, q0, q1, ws)
    return out


CELL = ("fcc", 6, 3, 4, 4.0, (32, 32, 32))


def test_direct_stages_leave_the_workspace_as_it_is(bse):
    plan, inf, ws = _prepare(bse, *CELL)
    before = torch.view_as_real(ws).view(torch.int32).clone()
    for flags in (bse.BSE_PD_DIRECT, bse.BSE_PD_DIRECT | bse.BSE_PD_TENSOR):
        _direct(bse, plan, inf, ws, 0, inf["nq"], flags)
        bse.bse_status_read(plan)
        assert torch.equal(torch.view_as_real(ws).view(torch.int32), before)


def test_ranges_on_two_streams_share_a_workspace(bse):
    plan, inf, ws = _prepare(bse, *CELL)
    ranges = [(0, 36), (36, 108), (108, 180), (180, 216)]
    ref = [_direct(bse, plan, inf, ws, a, b, bse.BSE_PD_DIRECT).clone() for a, b in ranges]
    outs = [torch.empty_like(r) for r in ref]
    streams = [torch.cuda.Stream() for _ in ranges]
    torch.cuda.synchronize()
    for _ in range(10):
        for o in outs:
            o.zero_()
        torch.cuda.synchronize()
        for st, (a, b), o in zip(streams, ranges, outs):
            with torch.cuda.stream(st):
                _direct(bse, plan, inf, ws, a, b, bse.BSE_PD_DIRECT, o)
        torch.cuda.synchronize()
        bse.bse_status_read(plan)
        for o, r in zip(outs, ref):
            assert torch.equal(o, r)


# tiles: 20,736 (odd ranges of a sheet); 216,000, more than one launch holds; a prime mesh with regions of one point
@pytest.mark.parametrize("n,nv,nc,ranges", [(24, 1, 2, [(0, 576), (23, 24), (100, 333), (575, 576)]),
                                            (60, 1, 1, [(0, 1), (1777, 1811), (3590, 3600)]),
                                            (23, 2, 3, [(0, 40), (511, 529)])])
def test_tiles_of_any_range(bse, n, nv, nc, ranges):
    plan, inf, ws = _prepare(bse, "hex", n, nv, nc, 2.5, (12, 12, 48))
    tol = 2.0 ** -21 + 24 * 2.0 ** -23 + (inf["tc_kpad"] / 32 + 4 * inf["tc_kpad"]) * 2.0 ** -24
    for q0, q1 in ranges:
        bse.bse_set_pair_variant(plan, 0, -1)
        t = _direct(bse, plan, inf, ws, q0, q1, bse.BSE_PD_DIRECT | bse.BSE_PD_TENSOR)
        bse.bse_set_pair_variant(plan, 0, 64)
        p = _direct(bse, plan, inf, ws, q0, q1, bse.BSE_PD_DIRECT)
        bse.bse_status_read(plan)
        assert float((t - p).abs().max()) <= tol and float(t.abs().max()) > 0.0, (q0, q1)
