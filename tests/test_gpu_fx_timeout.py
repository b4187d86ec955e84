"""Failure detection of the fixed-point marches' bounded waits, made to happen on purpose without
faulting anything: the test hook (swr_test_wait_hook) makes one subdomain hand nothing on, with a
short limit.  The waits for the rows of a cluster, or for a step's factors (V(t,x): one warp,
several warps of one CTA, a cluster), run out, the march leaves as a whole and the call reports
SWR_ERR_TIMEOUT.  The context stays usable: with the hook cleared a fresh plan marches right."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1503_02564_gb300 import workloads as W
from test_gpu_fixed_point_paths import TOL_MARCH, dev, moving, problem, rel, workload

pytestmark = pytest.mark.gpu

CASES = {   # (chunk, sizes, V(t,x), the list that waits)
    "cluster": (12, [4121, 2000, 4000], False, "build"),
    "streamed one warp": (4, [140, 150, 145], True, "zero_flux"),
    "streamed several warps": (4, [400, 390, 410], True, "zero_flux"),
    "streamed cluster": (8, [3300, 3000, 3100], True, "zero_flux"),
}


def plan_of(swr, wl, chunk):
    return swr.Plan(nx=wl.nx, a0=wl.a0, b0=wl.b0, nt=wl.nt, dt=wl.dt, nsub=wl.nsub, node_off=wl.off,
                    p=wl.sigma, vkind=swr.SWR_V_TIME if wl.V.ndim == 2 else swr.SWR_V_STATIC,
                    tuning={"chunk_L": chunk, "autotune": -1})


@pytest.mark.parametrize("case", sorted(CASES))
def test_withheld_rows_time_out_and_the_device_recovers(case):
    from paper_1503_02564_gb300 import swr
    chunk, sizes, timed, name = CASES[case]
    wl = workload(sizes, 80)
    if timed:
        wl = moving(wl)
    V, u0 = dev(wl.V), dev(wl.u0)
    plan = plan_of(swr, wl, chunk)
    try:
        swr.swr_test_wait_hook(5000, 1)
        with pytest.raises(swr.SWRError) as e:
            plan.build_interface(V, u0)
        assert e.value.status == swr.SWR_ERR_TIMEOUT
        # the subdomain's systems are flagged, the others are not
        n, again = plan.fixed_point_counts()[name]
        assert n > 0 and again == (3 if name == "build" else 1)
    finally:
        swr.swr_test_wait_hook(0, -1)
        plan.destroy()
    plan = plan_of(swr, wl, chunk)
    plan.build_interface(V, u0)
    assert plan.fixed_point_counts()[name] == (n, 0)
    d = torch.zeros(plan.n_interface, dtype=torch.complex128, device="cuda")
    plan.get_interface(d, None)
    plan.destroy()
    assert rel(d.cpu().numpy(), O.build_d(problem(wl))) < TOL_MARCH
