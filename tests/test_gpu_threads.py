"""Two host threads, each with its own stream, system and buffers, whose calls launch the same kernels with different
amounts of shared memory: a limit that one thread sets must not refuse the other's launch.
"""
import threading

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


def _rand(gen, *shape):
    return torch.view_as_complex(torch.randn(*shape, 2, generator=gen, device="cuda"))


def _run(jobs, reps):
    errors = []

    def work(job):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(reps):
                    job()
                torch.cuda.current_stream().synchronize()
        except Exception as e:  # noqa: BLE001
            errors.append(e)
    torch.cuda.synchronize()
    threads = [threading.Thread(target=work, args=(j,)) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors


def test_block_products_of_two_systems(bse):
    jobs, checks = [], []
    for i, (nv, nc) in enumerate(((3, 3), (3, 4))):
        plan = bse.Plan([SystemSpec("cell", "fcc", 10.0, 0.0, (2, 2, 2), nv, nc, 1.6, (24,) * 3, "3d")])
        inf = plan.info(0)
        gen = torch.Generator(device="cuda").manual_seed(3 + i)
        rho = _rand(gen, bse.bse_rho_dir_count(plan, 0, 0, inf["nq"]), inf["ng_max"])
        W = _rand(gen, inf["nq"], inf["ng_max"], inf["ng_max"])
        W = (W + W.mH).contiguous()
        H = torch.zeros(inf["dim"], inf["dim"], dtype=torch.complex64, device="cuda")
        ws = torch.empty(bse.bse_workspace_size(plan, 0, bse.BSE_WS_KERNEL, inf["nq"]) // 8 + 1, dtype=torch.complex64,
                         device="cuda")

        def job(plan=plan, inf=inf, rho=rho, W=W, H=H, ws=ws):
            H.zero_()
            bse.bse_build_kernel(plan, 0, bse.BSE_BK_DIRECT, None, rho, 0, inf["nq"], W, None, 0.0, bse.BSE_PREC_FP32, H, ws)
        job()
        jobs.append(job)
        checks.append((H, H.clone(), plan))
    _run(jobs, 400)
    for H, ref, plan in checks:
        assert torch.equal(H, ref)
        bse.bse_status_read(plan)


def test_dyson_of_two_sizes(bse):
    jobs, checks = [], []
    for ecut in (1.0, 8.0):
        plan = bse.Plan([SystemSpec("cell", "fcc", 10.0, 0.0, (2, 2, 2), 1, 1, ecut, (32,) * 3, "3d")])
        n, nw = plan.info(0)["ng0"], 4
        gen = torch.Generator(device="cuda").manual_seed(n)
        chi = (_rand(gen, nw, n, n) * (0.1 / np.sqrt(n))).contiguous()
        eps = torch.zeros(nw, dtype=torch.complex128, device="cuda")
        ws = torch.empty(bse.bse_workspace_size(plan, 0, bse.BSE_WS_EPSM, nw) // 8 + 1, dtype=torch.complex64, device="cuda")

        def job(plan=plan, chi=chi, eps=eps, ws=ws):
            bse.bse_epsilon_macro(plan, 0, chi, None, eps, ws)
        job()
        torch.cuda.synchronize()
        jobs.append(job)
        checks.append((eps, eps.clone()))
    _run(jobs, 200)
    for eps, ref in checks:
        assert torch.equal(eps, ref)
