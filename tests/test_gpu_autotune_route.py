"""Tuning a system whose direct set takes the tensor cores by default: the tuner times that form against the variants and the
plan keeps the faster, also from a cache and from an entry of before it was a candidate; tensor_choice holds in both
precisions."""
import json

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


def test_tuned_system_keeps_the_faster_route(bse, tmp_path):
    from paper_1206_3518_gb300 import autotune
    from paper_1206_3518_gb300.pipeline import Forward
    spec = SystemSpec("tune", "fcc", 10.0, 0.0, (6, 6, 6), 3, 4, 4.0, (32,) * 3, "3d")
    s = generate(spec, wdtype=np.complex64)
    coef = torch.as_tensor(s.coef, dtype=torch.complex64, device="cuda")
    en = torch.as_tensor(s.energies, dtype=torch.float64, device="cuda")
    W = torch.as_tensor(s.W, dtype=torch.complex64, device="cuda")
    plan = bse.Plan([spec])
    F = Forward(plan, 0, nsteps=8, nw=8)
    nq = F.nq
    assert bse.bse_pair_route(plan, 0, 0, nq)
    untuned = F.build(coef, en, W, spec.delta).clone()
    cache = str(tmp_path / "tune.json")
    r = autotune.tune(plan, 0, F, cache_path=cache)
    route = bse.bse_pair_route(plan, 0, 0, nq)
    t_tensor = autotune._time_tensor(plan, 0, F, 0, nq, 3)
    t_best = r["ms"][str(r["variant"]["index"])]
    if not 0.8 < t_tensor / t_best < 1.25:             # far enough apart for two timings to agree
        assert route == (t_tensor < t_best)
    if route:
        assert torch.equal(F.build(coef, en, W, spec.delta), untuned)
    plan2 = bse.Plan([spec])
    assert autotune.tune(plan2, 0, F, cache_path=cache)["cached"]
    assert bse.bse_pair_route(plan2, 0, 0, nq) == route
    stored = json.load(open(cache))
    for e in stored.values():
        del e["default_tensor"]
    json.dump(stored, open(cache, "w"))
    plan3 = bse.Plan([spec])
    assert autotune.tune(plan3, 0, F, cache_path=cache)["cached"] and bse.bse_pair_route(plan3, 0, 0, nq)
    r = autotune.tune(plan3, 0, F, cache_path=cache, with_tensor=True)
    assert bse.bse_pair_route(plan3, 0, 0, nq) == r["tensor"] == F.tensor_choice
