"""V-cycles and solves at fixed Chebyshev degrees against the oracle.  Degree 1 takes single
steps on level 0; from 2 on the first two steps are one pass, from 3 on a pass that also leaves the
direction for the next step.  Tolerances are those of the degree-2 tests: 1e-11 of the largest
entry for an FP64 V-cycle, 2e-5 for FP32, 1e-10 and one iteration for an FP64 solve."""
import numpy as np
import pytest

from paper_0907_4863_gb300 import inputs as I
from tests.oracle_cases import oracle_hierarchy, oracle_operator

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    import torch
    from paper_0907_4863_gb300 import build
    build.build()
    from paper_0907_4863_gb300 import saamg
    assert torch.cuda.is_available()
    torch.cuda.set_device(0)
    saamg.use_torch_allocator()
    return saamg


WORKLOADS = [(I.pipe_workload(40, I.QUADRATIC), dict(max_coarse=150)),
             (I.taper_workload(33, 30, 47, I.LINEAR), dict(max_coarse=100))]


@pytest.mark.parametrize("degree", [1, 2, 3, 4])
@pytest.mark.parametrize("prec", [0, 1], ids=["fp64", "fp32"])
@pytest.mark.parametrize("w,prm", WORKLOADS, ids=lambda v: getattr(v, "name", ""))
def test_vcycle_and_solve_at_degree(S, w, prm, prec, degree):
    import torch
    o = oracle_operator(w)
    oh = oracle_hierarchy(o, cheb_degree=degree, **prm)
    op = S.build_operator(S.make_domain(w.domain), S.make_grid(w.grid), w.mode)
    h = S.setup(op, S.params_default(cheb_degree=degree, precision=prec, beta_rule=1, **prm))
    r = np.random.default_rng(17).standard_normal(o.n)
    ref = oh.vcycle(r)
    buf = torch.zeros(o.n + 1, dtype=torch.float64, device="cuda")
    for at in (0, 1):  # the caller's vector on a 16-byte boundary and off it
        z = torch.empty(o.n, dtype=torch.float64, device="cuda")
        x = buf[at:at + o.n]
        x.copy_(torch.from_numpy(r))
        S.vcycle(h, x, z)
        err = np.max(np.abs(z.cpu().numpy() - ref)) / np.max(np.abs(ref))
        assert err < (1e-11 if prec == 0 else 2e-5), (at, err)
    rho = I.gaussian_bunch(w.grid, w.centre, w.sigma, 18)
    phi_ref, oinfo = oh.solve(rho, rtol=1e-8, beta_rule=1)
    phi = torch.zeros(w.grid.nbox, dtype=torch.float64, device="cuda")
    info = S.solve(h, torch.from_numpy(rho).cuda(), phi, rtol=1e-8)
    assert info["converged"] == 1 and info["relres_true"] <= 1.5e-8
    assert abs(info["iters"] - oinfo["iters"]) <= (1 if prec == 0 else 2)
    if prec == 0:
        assert np.max(np.abs(phi.cpu().numpy() - phi_ref)) <= 1e-10 * np.max(np.abs(phi_ref))
    h.free()
    op.free()
