"""Paths of the fixed-point marches that only some systems of a plan take, each shown to be taken
by the plan's counts: systems marched again in FP64 next to systems that stay in fixed point
(factors out of range, cross responses too small, states that grow too fast), u(T) superposed from
both kinds of records, and the streamed marches (V(t,x)) over clusters, with a step out of
range, with growing fluxes.  Against the oracle's marches to the march tolerance of the other
tests (relative L2 1e-10), and its solve to 1e-9."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1503_02564_gb300 import workloads as W

pytestmark = pytest.mark.gpu
TOL_MARCH, TOL_SOLVE = 1e-10, 1e-9


def rel(a, b):
    return float(np.linalg.norm(np.ravel(a) - np.ravel(b)) / max(np.linalg.norm(np.ravel(b)), 1e-300))


def workload(sizes, nt, h=5e-4, p=None, inside=None, value=0.0):
    """Subdomains of the given numbers of elements, a wave of size one everywhere; the potential
    of subdomain `inside` raised by `value`, smoothly, away from its ends."""
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int32)
    nx = int(off[-1]) + 1
    half = 0.5 * h * (nx - 1)
    x = np.linspace(-half, half, nx)
    V = -4.0 * np.exp(-x * x / 2)
    if inside is not None:
        a, b = off[inside], off[inside + 1]
        s = np.arange(b - a + 1) / (b - a)
        V[a:b + 1] += value * np.clip(8 * np.minimum(s, 1 - s), 0, 1) ** 2
    wl = W.Workload("fx", -half, half, nx, 1e-3, nt, off, V, np.exp(3j * x) * (1.0 + 0.3 * np.sin(0.7 * x)))
    if p is not None:
        wl.sigma = p
    return wl


def problem(wl, tc=0):
    return O.Problem(wl.a0, wl.b0, wl.nx, wl.dt, wl.nt, wl.off.astype(np.int64), wl.u0, wl.V,
                     tc=tc, sigma=wl.sigma, vkind=O.V_TIME if wl.V.ndim == 2 else O.V_STATIC)


def dev(a):
    return torch.tensor(np.ravel(a), device="cuda")


def make(wl, chunk=0, tc=0, **kw):
    from paper_1503_02564_gb300 import swr
    plan = swr.Plan(nx=wl.nx, a0=wl.a0, b0=wl.b0, nt=wl.nt, dt=wl.dt, nsub=wl.nsub, node_off=wl.off,
                    p=wl.sigma, tc=tc, vkind=swr.SWR_V_TIME if wl.V.ndim == 2 else swr.SWR_V_STATIC,
                    tuning={"chunk_L": chunk, "autotune": -1}, **kw)
    plan.build_interface(dev(wl.V), dev(wl.u0))
    return plan


def interface(plan):
    d = torch.zeros(plan.n_interface, dtype=torch.complex128, device="cuda")
    cols = torch.zeros(plan.n_cols, dtype=torch.complex128, device="cuda")
    plan.get_interface(d, cols)
    return d.cpu().numpy(), cols.cpu().numpy()


def apply_R(plan, g):
    gi = dev(g)
    go = torch.zeros_like(gi)
    plan.apply_R(gi, go)
    return go.cpu().numpy()


# V = 1e6: couplings above one within a chunk, factors out of range.  V = -20000: nothing crosses
# (1e-12 over 0.4): the impulses' cross responses are below 2^-16 of their state.
@pytest.mark.parametrize("value,again", [(1e6, 3), (-20000.0, 2)])
@pytest.mark.parametrize("chunk,sizes", [(12, [400, 400, 800, 390]),      # one warp a system, and two
                                         (4, [800, 2000, 1900, 2000])])   # 161 to 401 separators
def test_some_systems_again(value, again, chunk, sizes):
    from paper_1503_02564_gb300 import swr
    wl = workload(sizes, 80, inside=2 if chunk == 12 else 1, value=value)
    plan = make(wl, chunk, precond=swr.SWR_PC_CAUSAL)
    d, cols = interface(plan)
    systems, bad = plan.fixed_point_counts()["build"]
    assert systems == 3 * wl.nsub - 2 and bad == again
    g = W.random_interface(wl.nblk, wl.nt, 61)
    r = apply_R(plan, g)
    assert plan.fixed_point_counts()["R"][0] == wl.nsub
    P = problem(wl)
    assert rel(d, O.build_d(P)) < TOL_MARCH
    assert rel(cols, O.build_columns(P)) < TOL_MARCH
    assert rel(r, O.apply_R(P, g)) < TOL_MARCH
    # u(T) superposed from integer states and, for the flagged systems, from FP64 ones; the second
    # solve after a build replayed from the graph
    gs, uTm = O.mono_interface(P)
    for _ in range(3):
        uT = torch.zeros(wl.nx, dtype=torch.complex128, device="cuda")
        gx = torch.zeros(plan.n_interface, dtype=torch.complex128, device="cuda")
        plan.solve(gx, False, uT)
        assert rel(uT.cpu().numpy(), uTm) < TOL_SOLVE and rel(gx.cpu().numpy(), gs) < TOL_SOLVE
        plan.build_interface(dev(wl.V), dev(wl.u0))
    assert plan.get_stats()["superposed"] == 1
    plan.destroy()


def test_some_systems_again_in_a_batch():
    from paper_1503_02564_gb300 import swr
    wls = [workload([400, 800, 390], 60, inside=1, value=1e6), workload([700, 410, 1500], 80),
           workload([400, 800, 390], 70, inside=1, value=-20000.0)]
    plan = swr.BatchPlan([dict(nx=w.nx, a0=w.a0, b0=w.b0, nt=w.nt, nsub=w.nsub, node_off=w.off) for w in wls],
                         dt=1e-3, p=wls[0].sigma, precond=swr.SWR_PC_CAUSAL,
                         tuning={"chunk_L": 12, "autotune": -1})
    plan.build_interface(dev(np.concatenate([w.V for w in wls])), dev(np.concatenate([w.u0 for w in wls])))
    assert plan.fixed_point_counts()["build"] == (21, 5)
    d, cols = interface(plan)
    uT = torch.zeros(plan.nx, dtype=torch.complex128, device="cuda")
    plan.solve(None, False, uT)
    uT = uT.cpu().numpy()
    kb = kc = ku = 0
    for w in wls:
        P = problem(w)
        ref, rc = O.build_d(P), O.build_columns(P)
        assert rel(d[kb:kb + np.size(ref)], ref) < TOL_MARCH
        assert rel(cols[kc:kc + np.size(rc)], rc) < TOL_MARCH
        assert rel(uT[ku:ku + w.nx], O.mono_interface(P)[1]) < TOL_SOLVE
        kb, kc, ku = kb + np.size(ref), kc + np.size(rc), ku + w.nx
    plan.destroy()


def test_growth_goes_back_to_fp64():
    """Robin ends with gain: the states grow fourfold a step, faster than they are scaled down."""
    wl = workload([400, 390, 800], 60, p=-24.5 + 24.5j)
    plan = make(wl, 12)
    systems, bad = plan.fixed_point_counts()["build"]
    assert systems == 7 and bad > 0
    d, cols = interface(plan)
    plan.destroy()
    P = problem(wl)
    assert rel(d, O.build_d(P)) < TOL_MARCH and rel(cols, O.build_columns(P)) < TOL_MARCH


# ---- V(t,x): per-step factors ------------------------------------------------------------
def moving(wl, at=None):
    """V(t,x) from the workload's potential; `at` = (row, subdomain, value): raised in one row."""
    t = np.arange(wl.nt + 1)[:, None] * wl.dt
    V = wl.V[None, :] * (1.0 + 0.5 * np.sin(40.0 * t))
    if at:
        V[at[0], wl.off[at[1]] + 1:wl.off[at[1] + 1]] += at[2]
    wl.V = V
    return wl


def check_streamed(wl, chunk, counts, g=None, **kw):
    plan = make(wl, chunk)
    if g is None:
        g = W.random_interface(wl.nblk, wl.nt, 62)
    d, _ = interface(plan)
    assert plan.fixed_point_counts()["zero_flux"] == (wl.nsub, counts)
    r = apply_R(plan, g)
    n, again = plan.fixed_point_counts()["R"]
    assert n == wl.nsub and again == counts
    plan.destroy()
    P = problem(wl)
    assert rel(d, O.build_d(P)) < TOL_MARCH
    assert rel(r, O.apply_R(P, g)) < TOL_MARCH


@pytest.mark.parametrize("chunk", [4, 8])
@pytest.mark.parametrize("seps", [31, 32, 33, 63, 64, 65])
def test_streamed_separator_counts(chunk, seps):
    full = (seps - 1) * (chunk + 1)
    check_streamed(moving(workload([full, full - 3, full - chunk, full], 40)), chunk, 0)


@pytest.mark.parametrize("chunk,sizes", [(4, [1700, 2400, 4700]),      # 341, 481 and 941 separators
                                         (8, [3300, 31 * 9, 8800]),    # 368, 32 and 979
                                         (8, [2304, 2295, 1152])])     # 257, 256 and 129
def test_streamed_clusters(chunk, sizes):
    check_streamed(moving(workload(sizes, 40)), chunk, 0)


@pytest.mark.parametrize("sizes", [[400, 390, 410], [2000, 1990, 2010]])
def test_streamed_step_out_of_range(sizes):
    check_streamed(moving(workload(sizes, 40), (20, 1, 4e6)), 4, 1)


@pytest.mark.parametrize("chunk,sizes", [(4, [400, 390, 1200]), (8, [200, 3300, 900])])
def test_streamed_state_scaled_down(chunk, sizes):
    wl = moving(workload(sizes, 64))
    g = W.random_interface(wl.nblk, wl.nt, 52) * (2.0 ** (40.0 * np.arange(wl.nt) / wl.nt))
    check_streamed(wl, chunk, 0, g)


# ---- factors within the range ------------------------------------------------------------
@pytest.mark.parametrize("nx,h,nt,nsub", [(1355, 24 / 1354, 372, 4), (862, 1.6e-2, 150, 3),
                                          (1700, 24 / 1699, 300, 5), (278, 24 / 277, 473, 6),
                                          (420, 24 / 419, 400, 6)])
@pytest.mark.parametrize("chunk", [0, 4, 8, 12])
def test_coarse_grids_stay_in_fixed_point(nx, h, nt, nsub, chunk):
    """Grids on which the chunks' solutions are largest against their right-hand sides."""
    base, extra = divmod(nx - 1, nsub)
    wl = workload([base + (j < extra) for j in range(nsub)], nt, h)
    wl.V = -wl.x ** 2 / 4
    plan = make(wl, chunk)
    d, cols = interface(plan)
    assert plan.fixed_point_counts()["build"] == (3 * nsub - 2, 0)
    r = apply_R(plan, W.random_interface(wl.nblk, wl.nt, 63))
    assert plan.fixed_point_counts()["R"] == (nsub, 0)
    plan.destroy()
    P = problem(wl)
    assert rel(d, O.build_d(P)) < TOL_MARCH and rel(cols, O.build_columns(P)) < TOL_MARCH
    assert rel(r, O.apply_R(P, W.random_interface(wl.nblk, wl.nt, 63))) < TOL_MARCH


# ---- nothing of the build is put off -----------------------------------------------------
@pytest.mark.parametrize("nx,nsub", [(48015, 80), (22190, 3), (20543, 11), (159333, 18)])
@pytest.mark.parametrize("tc", [0, 1])
def test_first_march_after_a_build_is_like_the_next(nx, nsub, tc):
    """R g launches the same kernels right after a build as later: the build has formed its factors."""
    from paper_1503_02564_gb300 import swr
    base, extra = divmod(nx - 1, nsub)
    wl = workload([base + (j < extra) for j in range(nsub)], 40)
    plan = swr.Plan(nx=wl.nx, a0=wl.a0, b0=wl.b0, nt=wl.nt, dt=wl.dt, nsub=wl.nsub, node_off=wl.off,
                    p=wl.sigma, tc=tc)
    g = W.random_interface(wl.nblk, wl.nt, 64)
    launches, out = [], []
    for k in range(4):
        if k < 3:
            plan.build_interface(dev(wl.V * (1.0 + min(k, 1))), dev(wl.u0))
        n0 = swr.swr_kernel_launch_count()
        out.append(apply_R(plan, g))
        launches.append(swr.swr_kernel_launch_count() - n0)
    plan.destroy()
    # (where R g has a chunk length of its own, the plan's very first march of it forms the factors)
    assert launches[0] >= launches[1] == launches[2] == launches[3]
    assert np.array_equal(out[1], out[2]) and np.array_equal(out[2], out[3])
    wl.V = wl.V * 2.0
    assert rel(out[1], O.apply_R(problem(wl, tc), g)) < TOL_MARCH


# ---- lists that are faster in FP64 -------------------------------------------------------
def test_list_with_flagged_systems_settles_in_fp64():
    """One subdomain of eight out of range: the second march, which only starts when the others
    are done, takes the build past its time in FP64 (4.5 against 2.9 ms), so the first build
    settles on FP64.  Later builds (the third is replayed from the graph) and solves agree."""
    from paper_1503_02564_gb300 import swr
    wl = workload([2500] * 8, 200, inside=3, value=1e6)
    plan = swr.Plan(nx=wl.nx, a0=wl.a0, b0=wl.b0, nt=wl.nt, dt=wl.dt, nsub=wl.nsub, node_off=wl.off,
                    p=wl.sigma, precond=swr.SWR_PC_CAUSAL)
    P = problem(wl)
    dr, cr, (gs, uTm) = O.build_d(P), O.build_columns(P), O.mono_interface(P)
    g = W.random_interface(wl.nblk, wl.nt, 65)
    rr = O.apply_R(P, g)
    for k in range(3):
        plan.build_interface(dev(wl.V), dev(wl.u0))
        assert plan.fixed_point_counts()["build"] == (0, 0)
        d, cols = interface(plan)
        uT = torch.zeros(wl.nx, dtype=torch.complex128, device="cuda")
        gx = torch.zeros(plan.n_interface, dtype=torch.complex128, device="cuda")
        plan.solve(gx, False, uT)
        assert rel(d, dr) < TOL_MARCH and rel(cols, cr) < TOL_MARCH
        assert rel(apply_R(plan, g), rr) < TOL_MARCH
        assert rel(uT.cpu().numpy(), uTm) < TOL_SOLVE and rel(gx.cpu().numpy(), gs) < TOL_SOLVE
    assert plan.get_stats()["superposed"] == 1
    plan.destroy()


def test_streamed_list_with_flagged_systems_settles_in_fp64():
    from paper_1503_02564_gb300 import swr
    wl = moving(workload([400, 390, 410], 40), (20, 1, 4e6))
    plan = swr.Plan(nx=wl.nx, a0=wl.a0, b0=wl.b0, nt=wl.nt, dt=wl.dt, nsub=wl.nsub, node_off=wl.off,
                    p=wl.sigma, vkind=swr.SWR_V_TIME)
    P = problem(wl)
    g = W.random_interface(wl.nblk, wl.nt, 66)
    for k in range(3):
        plan.build_interface(dev(wl.V), dev(wl.u0))
        assert plan.fixed_point_counts()["zero_flux"] == (0, 0)
        assert rel(interface(plan)[0], O.build_d(P)) < TOL_MARCH
        assert rel(apply_R(plan, g), O.apply_R(P, g)) < TOL_MARCH
        assert plan.fixed_point_counts()["R"] == (0, 0)
    plan.destroy()
