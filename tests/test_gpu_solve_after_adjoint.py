"""swr_solve needs no new build after swr_adjoint: the gradient's own zero-flux march leaves the
states that the build recorded for u(T) as they are.  The second solve repeats the first one's
arithmetic on the same data, so that u(T) and g are equal bit for bit; with the fixed-point and
with the FP64 marches, Robin and S_0^2 ends."""
import numpy as np
import pytest
import torch

from paper_1503_02564_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("two_level", [0, -1])
@pytest.mark.parametrize("tc", [0, 1])
def test_solve_after_adjoint(two_level, tc):
    from paper_1503_02564_gb300 import swr
    wl = W.config2(nsub=8, nx=4001, nt=40)
    plan = swr.Plan(nx=wl.nx, a0=wl.a0, b0=wl.b0, nt=wl.nt, dt=wl.dt, nsub=wl.nsub, node_off=wl.off,
                    p=wl.sigma, tc=tc, precond=swr.SWR_PC_CAUSAL, tuning={"two_level": two_level})
    plan.build_interface(torch.tensor(wl.V, device="cuda"), torch.tensor(wl.u0, device="cuda"))
    out = []
    for k in range(2):
        uT = torch.zeros(wl.nx, dtype=torch.complex128, device="cuda")
        g = torch.zeros(plan.n_interface, dtype=torch.complex128, device="cuda")
        plan.solve(g, False, uT)
        out.append((uT.cpu().numpy(), g.cpu().numpy()))
        if k == 0:
            assert plan.get_stats()["superposed"] == 1
            ubar = torch.empty_like(uT)
            plan.misfit(uT, torch.tensor(wl.u0 * np.exp(0.4j), device="cuda"), ubar)
            plan.adjoint(ubar, torch.empty(wl.nx, dtype=torch.float64, device="cuda"), 10)
    plan.destroy()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
