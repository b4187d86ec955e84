"""The fixed-point marches hold FP64's accuracy where the factors' own rounding does not cover
theirs: on coarse grids (dt/h^2 of order one), against the extended-precision build.

Bound: the error may be 1.4 times that of the FP64 marches at the same chunk length (both are
rounding errors of some hundred steps, the same in mean; two marches of FP64 that differ in chunk
length alone differ by up to a third).  S_0^2 ends march in FP64 on such grids."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1503_02564_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def outputs(wl, chunk, two_level, tc=0, time=False):
    from paper_1503_02564_gb300 import swr
    plan = swr.Plan(nx=wl.nx, a0=wl.a0, b0=wl.b0, nt=wl.nt, dt=wl.dt, nsub=wl.nsub, node_off=wl.off,
                    p=wl.sigma, tc=tc, vkind=swr.SWR_V_TIME if time else swr.SWR_V_STATIC,
                    tuning={"chunk_L": chunk, "autotune": -1, "two_level": two_level})
    V = np.tile(wl.V, wl.nt + 1) if time else wl.V
    plan.build_interface(torch.tensor(V, device="cuda"), torch.tensor(wl.u0, device="cuda"))
    d = torch.zeros(plan.n_interface, dtype=torch.complex128, device="cuda")
    cols = torch.zeros(plan.n_cols, dtype=torch.complex128, device="cuda")
    plan.get_interface(d, cols)
    plan.destroy()
    return d.cpu().numpy(), cols.cpu().numpy()


def workload(sizes, nt, h):
    nx = int(sum(sizes)) + 1
    half = 0.5 * h * (nx - 1)
    x = np.linspace(-half, half, nx)
    return W.Workload("coarse", -half, half, nx, 1e-3, nt,
                      np.concatenate([[0], np.cumsum(sizes)]).astype(np.int32), -x * x / 4,
                      np.exp(-(x - 0.4) ** 2 / 2 + 5j * x))


def error(a, x):
    return float(np.linalg.norm((np.asarray(a, np.clongdouble).ravel() - np.ravel(x)).astype(np.complex128)))


@pytest.mark.parametrize("chunk,sizes,h", [(8, [250, 250, 250, 250], 2.4e-2),    # one warp a system
                                           (4, [250, 240, 245, 250], 2.4e-2),    # 51 separators
                                           (8, [300, 310, 290], 1.2e-2)])
def test_coarse_grid(chunk, sizes, h):
    wl = workload(sizes, 200, h)
    P = O.Problem(wl.a0, wl.b0, wl.nx, wl.dt, wl.nt, wl.off.astype(np.int64), wl.u0, wl.V, sigma=wl.sigma)
    dx, cx, _, _ = O.build_ext(P)
    d1, c1 = outputs(wl, chunk, 0)
    d0, c0 = outputs(wl, chunk, -1)
    assert not np.array_equal(c1, c0)          # two ways of marching
    assert error(c1, cx) <= 1.4 * error(c0, cx)
    assert error(d1, dx) <= 1.4 * error(d0, dx)


@pytest.mark.parametrize("chunk", [4, 8])
def test_coarse_grid_streamed(chunk):
    """Per-step factors (the same potential in every row of V(t,x))."""
    wl = workload([250, 240, 250], 200, 2.4e-2)
    P = O.Problem(wl.a0, wl.b0, wl.nx, wl.dt, wl.nt, wl.off.astype(np.int64), wl.u0, wl.V, sigma=wl.sigma)
    dx, _, _, _ = O.build_ext(P)
    d1, _ = outputs(wl, chunk, 0, time=True)
    d0, _ = outputs(wl, chunk, -1, time=True)
    assert not np.array_equal(d1, d0)
    assert error(d1, dx) <= 1.4 * error(d0, dx)


def test_coarse_grid_s02():
    wl = workload([250, 250, 250, 250], 200, 2.4e-2)
    P = O.Problem(wl.a0, wl.b0, wl.nx, wl.dt, wl.nt, wl.off.astype(np.int64), wl.u0, wl.V, tc=1, sigma=wl.sigma)
    dx, cx, _, _ = O.build_ext(P)
    d1, c1 = outputs(wl, 8, 0, tc=1)
    d0, c0 = outputs(wl, 8, -1, tc=1)
    assert error(c1, cx) <= 1.4 * error(c0, cx)
    assert error(d1, dx) <= 1.4 * error(d0, dx)
