"""The fixed-point marches (csrc/swr_march_fx.cu) at the sizes where they can go wrong: separator
counts around the edges of a warp (31, 32, 33) and of a warp group of a cluster, uneven
subdomains in one launch, one and several CTAs per subdomain, driven marches whose state grows
and is scaled down on the way, and the cases that go back to FP64 (wrong-signed Robin
parameter, tiny cross responses, huge and zero data).  Against the oracle's marches to the
march tolerance of the other tests (relative L2 1e-10), and against the FP64 marches of the
same plan (tuning two_level = -1 keeps them) to 1e-12.
"""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1503_02564_gb300 import workloads as W

pytestmark = pytest.mark.gpu
TOL_MARCH = 1e-10


def rel(a, b):
    return float(np.linalg.norm(np.ravel(a) - np.ravel(b)) / max(np.linalg.norm(np.ravel(b)), 1e-300))


def workload(sizes, nt, h=5e-4, p=None):
    """Subdomains of the given numbers of elements, a wave of size one everywhere."""
    nx = int(sum(sizes)) + 1
    half = 0.5 * h * (nx - 1)
    x = np.linspace(-half, half, nx)
    wl = W.Workload("fx", -half, half, nx, 1e-3, nt, np.concatenate([[0], np.cumsum(sizes)]).astype(np.int32),
                    -4.0 * np.exp(-x * x / 2), np.exp(3j * x) * (1.0 + 0.3 * np.sin(0.7 * x)))
    if p is not None:
        wl.sigma = p
    return wl


def march(wl, chunk, two_level, g, tc=0):
    from paper_1503_02564_gb300 import swr
    plan = swr.Plan(nx=wl.nx, a0=wl.a0, b0=wl.b0, nt=wl.nt, dt=wl.dt, nsub=wl.nsub, node_off=wl.off,
                    p=wl.sigma, tc=tc, tuning={"chunk_L": chunk, "autotune": -1, "two_level": two_level})
    plan.build_interface(torch.tensor(wl.V, device="cuda"), torch.tensor(wl.u0, device="cuda"))
    d = torch.zeros(plan.n_interface, dtype=torch.complex128, device="cuda")
    cols = torch.zeros(plan.n_cols, dtype=torch.complex128, device="cuda")
    plan.get_interface(d, cols)
    gi = torch.tensor(g.ravel(), device="cuda")
    go = torch.zeros_like(gi)
    plan.apply_R(gi, go)
    plan.destroy()
    return d.cpu().numpy(), cols.cpu().numpy(), go.cpu().numpy()


def problem(wl, tc=0):
    return O.Problem(wl.a0, wl.b0, wl.nx, wl.dt, wl.nt, wl.off.astype(np.int64), wl.u0, wl.V,
                     tc=tc, sigma=wl.sigma)


def check(wl, chunk, g=None, against_f64=True):
    if g is None:
        g = W.random_interface(wl.nblk, wl.nt, 51)
    d1, c1, r1 = march(wl, chunk, 0, g)
    if against_f64:
        d0, c0, r0 = march(wl, chunk, -1, g)
        assert rel(d1, d0) < 1e-12 and rel(c1, c0) < 1e-12 and rel(r1, r0) < 1e-12
    P = problem(wl)
    assert rel(d1, O.build_d(P)) < TOL_MARCH
    assert rel(c1, O.build_columns(P)) < TOL_MARCH
    assert rel(r1, O.apply_R(P, g)) < TOL_MARCH


# P_j chunks of a subdomain of E elements with chunk length L: ceil(E / (L + 1)); P_j + 1 separators
@pytest.mark.parametrize("chunk", [4, 8, 12, 16])
@pytest.mark.parametrize("seps", [31, 32, 33, 63, 64, 65])
def test_separator_counts_around_a_warp(chunk, seps):
    full = (seps - 1) * (chunk + 1)
    check(workload([full, full - 3, full - chunk, full], 40), chunk)


@pytest.mark.parametrize("chunk,sizes", [
    (4, [2479, 2480, 2481, 2450]),          # 497, 497, 498, 491 separators, one and several CTAs
    (8, [31 * 9, 800, 3300, 64 * 9]),       # 32, 90, 368 and 65 separators in one launch
    (12, [415, 31 * 13, 4121, 95 * 13, 2000]),   # 33, 32, 318, 96, 155
    (16, [95 * 17, 31 * 17, 6001, 40]),     # 96, 32, 354 and 4 separators
])
def test_uneven_subdomains_over_clusters(chunk, sizes):
    check(workload(sizes, 130), chunk)


def test_short_chunks():
    """Subdomains so short that their chunks lack two and more of their nodes."""
    check(workload([2, 7, 30, 19, 14], 60, h=2e-2), 12)
    check(workload([3, 2, 5, 9], 60, h=5e-2), 8)


@pytest.mark.parametrize("chunk", [4, 12])
def test_driven_march_scales_its_state_down(chunk):
    """Fluxes that grow by 2^40 over the march: the state is scaled down on the way."""
    wl = workload([400, 390, 1200], 64)
    g = W.random_interface(wl.nblk, wl.nt, 52) * (2.0 ** (40.0 * np.arange(wl.nt) / wl.nt))
    check(wl, chunk, g)


@pytest.mark.parametrize("chunk,sizes", [
    (4, [150, 40, 155]), (8, [31 * 9, 800, 290]), (12, [400, 415, 2000]), (16, [31 * 17, 520, 3001])])
def test_s02_histories(chunk, sizes):
    """S_0^2 ends: the end histories as integer sums, over more steps than lanes.  The columns of
    an almost transparent condition are small differences of large terms (see test_gpu_long.py),
    so they are measured against the extended-precision build, relative to the summands, and
    the FP64 marches' distance to it is the yardstick for the plain errors."""
    wl = workload(sizes, 90)
    g = W.random_interface(wl.nblk, wl.nt, 51)
    d1, c1, r1 = march(wl, chunk, 0, g, 1)
    d0, c0, r0 = march(wl, chunk, -1, g, 1)
    P = problem(wl, 1)
    dx, cx, dm, cm = O.build_ext(P)
    for a, b, x, mag in ((d1, d0, dx, dm), (c1, c0, cx, cm)):
        e = np.linalg.norm((np.asarray(a, np.clongdouble).ravel() - np.ravel(x)).astype(np.complex128))
        f = np.linalg.norm((np.asarray(b, np.clongdouble).ravel() - np.ravel(x)).astype(np.complex128))
        assert e <= 1e-12 * np.linalg.norm(np.asarray(mag, np.float64).ravel())
        assert e <= 3.0 * f + 1e-14 * np.linalg.norm(np.asarray(mag, np.float64).ravel())
    assert rel(r1, r0) < 1e-11 and rel(r1, O.apply_R(P, g)) < TOL_MARCH


@pytest.mark.parametrize("scale", [0.0, 1e-270, 1e-150, 1e150])
def test_scales_of_the_data(scale):
    wl = workload([400, 390, 800], 40)
    wl.u0 = wl.u0 * scale
    check(wl, 12, W.random_interface(wl.nblk, wl.nt, 53) * scale, against_f64=scale > 1e-200)


def test_marches_that_go_back_to_fp64():
    # a Robin parameter with gain: the states grow without bound
    check(workload([400, 390, 800], 60, p=3.0 + 6.0j), 12, against_f64=False)
    # cross responses far below the impulse (no wave crosses in 20 steps)
    check(workload([3000, 3000, 3000], 20), 12)


def test_gradient_follows_a_new_potential():
    """A plan's second gradient, after a build with another potential, is the one of a fresh
    plan (its chunk length is not the build marches')."""
    from paper_1503_02564_gb300 import swr
    wl = workload([800, 790, 805], 40)
    tgt = torch.tensor(wl.u0 * np.exp(0.4j), device="cuda")
    out = []
    for Vs in ([1.0, 0.5], [0.5]):
        plan = swr.Plan(nx=wl.nx, a0=wl.a0, b0=wl.b0, nt=wl.nt, dt=wl.dt, nsub=wl.nsub,
                        node_off=wl.off, p=wl.sigma, precond=swr.SWR_PC_CAUSAL)
        for f in Vs:
            plan.build_interface(torch.tensor(wl.V * f, device="cuda"), torch.tensor(wl.u0, device="cuda"))
            uT = torch.zeros(wl.nx, dtype=torch.complex128, device="cuda")
            plan.solve(None, False, uT)
            ubar = torch.empty_like(uT)
            plan.misfit(uT, tgt, ubar)
            grad = torch.empty(wl.nx, dtype=torch.float64, device="cuda")
            plan.adjoint(ubar, grad, 10)
        out.append(grad.cpu().numpy())
        plan.destroy()
    assert rel(out[0], out[1]) < 1e-9


@pytest.mark.parametrize("chunk,sizes", [
    (12, [415, 31 * 13, 4121, 95 * 13, 2000, 64 * 13, 159 * 13]),   # 33, 32, 318, 96, 155, 65, 160 separators
    (4, [2479, 310 * 5, 7, 127 * 5, 128 * 5]),                      # 497, 311, 3, 128, 129
])
def test_batch_with_every_size_of_cluster(chunk, sizes):
    """Instances of uneven subdomains in one plan: one CTA, or a cluster of as many CTAs as the
    subdomain takes, one launch per shape.  Each instance is marched to 1e-10 of the oracle, and
    to 1e-12 of the FP64 marches of the same batch."""
    from paper_1503_02564_gb300 import swr
    wls = [workload(sizes, 130), workload(sizes[::-1], 100)]
    insts = [dict(nx=w.nx, a0=w.a0, b0=w.b0, nt=w.nt, nsub=w.nsub, node_off=w.off) for w in wls]
    gs = [W.random_interface(w.nblk, w.nt, 53 + k) for k, w in enumerate(wls)]
    out = []
    for two_level in (0, -1):
        plan = swr.BatchPlan(insts, dt=wls[0].dt, p=wls[0].sigma, tc=0,
                             tuning={"chunk_L": chunk, "autotune": -1, "two_level": two_level})
        plan.build_interface(torch.tensor(np.concatenate([w.V for w in wls]), device="cuda"),
                             torch.tensor(np.concatenate([w.u0 for w in wls]), device="cuda"))
        d = torch.zeros(plan.n_interface, dtype=torch.complex128, device="cuda")
        cols = torch.zeros(plan.n_cols, dtype=torch.complex128, device="cuda")
        plan.get_interface(d, cols)
        gi = torch.tensor(np.concatenate([g.ravel() for g in gs]), device="cuda")
        go = torch.zeros_like(gi)
        plan.apply_R(gi, go)
        plan.destroy()
        out.append([t.cpu().numpy() for t in (d, cols, go)])
    for a, b in zip(*out):
        assert rel(a, b) < 1e-12
    d, cols, go = out[0]
    kb = kc = 0
    for w, g in zip(wls, gs):
        P = problem(w)
        assert rel(d[kb:kb + g.size], O.build_d(P)) < TOL_MARCH
        assert rel(go[kb:kb + g.size], O.apply_R(P, g)) < TOL_MARCH
        ref = O.build_columns(P)
        assert rel(cols[kc:kc + np.size(ref)], ref) < TOL_MARCH
        kb, kc = kb + g.size, kc + np.size(ref)
