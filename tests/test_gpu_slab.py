"""GPU parity of the slab kernel (csrc/mg_slab.cu: the coarse part of the
V-cycle in one thread-block cluster) with the oracle and with the one-block
and per-phase launches, at sizes where its plan changes: one to three planes
per CTA, empty CTAs, tie (x_N = 1) and odd levels, the smallest level."""
import numpy as np
import pytest

from paper_2001_02327_gb300 import inputs as I
from tests.test_gpu_parity import gpu_solve, mg, omega, random_single_level, relmax  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,n", [(3, 4), (3, 7), (3, 8), (3, 9), (3, 16), (3, 17), (3, 31), (3, 32), (3, 33),
                                   (2, 6), (2, 22), (2, 23), (2, 64), (2, 127), (2, 158), (2, 159)])
@pytest.mark.parametrize("nu", [(1, 1), (3, 0), (0, 2)])
def test_fp64_slab_matches_oracle(mg, oracle, dim, n, nu):  # noqa: F811
    """Fixed-point V-cycles against the FP64 oracle after three cycles on
    random data (the parity bar of the FP64 path)."""
    H, inp = random_single_level(dim, n, 1000 * dim + n)
    _, g = gpu_solve(mg, H, inp, nu_pre=nu[0], nu_post=nu[1], max_cycles=3, rel_tol=0.0)
    ref = oracle.solve_hierarchy(H, inp, nu[0], nu[1], 3, 0.0)
    assert relmax(g[0]["phi"], omega(ref[0]["phi"], n, dim)) < 1e-12


@pytest.mark.parametrize("dim,n", [(3, 30), (2, 126), (2, 158)])
def test_fp64_slab_smooth_source_far_above_its_right_hand_side(mg, oracle, dim, n):  # noqa: F811
    """A constant density with a zero boundary: the potential is thousands of
    times the right-hand side h^2 f that fixes the first scale, so the scale
    has to give way during the ascent."""
    H = I.Hierarchy(dim, [n], [tuple([0.0] * dim)], 1.0 / n, 1.0, [], "const")
    inp = [{"rho": np.ones((n,) * dim), "bc_rho": np.ones((n + 2,) * dim), "bc_phi": np.zeros((n + 4,) * dim)}]
    _, g = gpu_solve(mg, H, inp, max_cycles=3, rel_tol=0.0)
    ref = oracle.solve_hierarchy(H, inp, 2, 1, 3, 0.0)
    assert relmax(g[0]["phi"], omega(ref[0]["phi"], n, dim)) < 1e-12


@pytest.mark.parametrize("scale", [1e-130, 1e-30, 1e130])
def test_fp64_slab_extreme_magnitudes(mg, scale):  # noqa: F811
    """The potential scales with the data over the whole range of exponents."""
    H, inp = random_single_level(3, 16, 5)
    big = [{k: v * scale for k, v in inp[0].items()}]
    _, a = gpu_solve(mg, H, inp, max_cycles=3, rel_tol=0.0)
    _, b = gpu_solve(mg, H, big, max_cycles=3, rel_tol=0.0)
    assert relmax(b[0]["phi"] / scale, a[0]["phi"]) < 1e-12


@pytest.mark.parametrize("dim,n", [(3, 16), (3, 33), (3, 47), (2, 64), (2, 127)])
@pytest.mark.parametrize("nu", [(2, 2), (1, 0), (0, 1)])
def test_fp32_slab_matches_phase_launches(mg, monkeypatch, dim, n, nu):  # noqa: F811
    """One FP32 correction step of two V-cycles in the slab kernel and as
    launches per phase differ by FP32 rounding only: some 50 dependent
    operations of 2^-24 each per cycle on a correction of the potential's own
    size, below 1e-5 of its largest value."""
    H, inp = random_single_level(dim, n, 77 + n)
    kw = dict(nu_pre=nu[0], nu_post=nu[1], max_cycles=2, rel_tol=0.0, precision=mg.MG_MIXED, inner_cycles=2)
    _, a = gpu_solve(mg, H, inp, **kw)
    monkeypatch.setenv("MG_BOTTOM_N32", "8")
    _, b = gpu_solve(mg, H, inp, **kw)
    assert relmax(a[0]["phi"], b[0]["phi"]) < 1e-5


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_fp64_slab_non_finite_density_reports_ediverged(mg, bad):  # noqa: F811
    H, inp = random_single_level(3, 16, 6)
    inp[0]["rho"][3, 4, 5] = bad
    with pytest.raises(mg.MGError) as ei:
        gpu_solve(mg, H, inp, max_cycles=5, rel_tol=1e-10)
    assert ei.value.status == mg.MG_EDIVERGED


@pytest.mark.parametrize("dim,n", [(3, 4), (3, 16), (3, 31), (3, 32), (2, 22), (2, 64), (2, 158)])
@pytest.mark.parametrize("max_cycles", [1, 30])
def test_fp64_slab_solve_stops_where_the_loop_of_launches_stops(mg, monkeypatch, dim, n, max_cycles):  # noqa: F811
    """A level solved by one launch takes the cycles that the loop of launches
    takes.  Residuals of potentials of order one round at 8 n^2 2^-53 of the
    right-hand side (12), below 2e-12 of it here."""
    H, inp = random_single_level(dim, n, 31 * n + dim)
    kw = dict(max_cycles=max_cycles, rel_tol=1e-8)
    _, a = gpu_solve(mg, H, inp, **kw)
    monkeypatch.setenv("MG_BOTTOM_N64", "8")
    _, b = gpu_solve(mg, H, inp, **kw)
    assert a[0]["cycles"] == b[0]["cycles"] and a[0]["status"] == b[0]["status"]
    assert abs(a[0]["rel_res"] - b[0]["rel_res"]) < 1e-11 * max(1.0, b[0]["rel_res"])
    assert relmax(a[0]["phi"], b[0]["phi"]) < 1e-12


def test_fp64_slab_solve_of_nothing(mg):  # noqa: F811
    """A zero right-hand side: no cycle, the zero potential."""
    n = 16
    H = I.Hierarchy(3, [n], [(0.0, 0.0, 0.0)], 1.0 / n, 1.0, [], "zero")
    inp = [{"rho": np.zeros((n,) * 3), "bc_rho": np.zeros((n + 2,) * 3), "bc_phi": np.zeros((n + 4,) * 3)}]
    _, g = gpu_solve(mg, H, inp, max_cycles=5, rel_tol=1e-10)
    assert g[0]["cycles"] == 0 and np.all(g[0]["phi"] == 0.0)


@pytest.mark.parametrize("dim,n", [(2, 20), (2, 22), (2, 23), (3, 5), (3, 7), (3, 8)])
@pytest.mark.parametrize("nu", [(2, 1), (1, 0)])
def test_fp64_slab_solve_of_a_level_in_one_cta(mg, monkeypatch, dim, n, nu):  # noqa: F811
    """Levels that CTA 0 holds alone (and the first that it does not), with a
    scale that gives way in the first ascent: every CTA of the cluster has to
    stop after the same cycle, the one where the loop of launches stops.  The
    residual of a potential of order one rounds below 1e-13 of the right-hand
    side at these sizes."""
    H = I.Hierarchy(dim, [n], [tuple([0.0] * dim)], 1.0 / n, 1.0, [], "const")
    inp = [{"rho": np.ones((n,) * dim), "bc_rho": np.ones((n + 2,) * dim), "bc_phi": np.zeros((n + 4,) * dim)}]
    kw = dict(nu_pre=nu[0], nu_post=nu[1], max_cycles=40, rel_tol=1e-8)
    _, a = gpu_solve(mg, H, inp, **kw)
    monkeypatch.setenv("MG_BOTTOM_N64", "8")
    _, b = gpu_solve(mg, H, inp, **kw)
    assert a[0]["cycles"] == b[0]["cycles"] and a[0]["status"] == b[0]["status"] == 0
    assert abs(a[0]["rel_res"] - b[0]["rel_res"]) < 1e-12
    assert relmax(a[0]["phi"], b[0]["phi"]) < 1e-12


@pytest.mark.parametrize("dim,n", [(3, 7), (3, 16), (3, 31), (2, 22), (2, 126)])
@pytest.mark.parametrize("nu", [(1, 0), (0, 1)])
def test_fp64_slab_solve_of_many_slow_cycles(mg, monkeypatch, dim, n, nu):  # noqa: F811
    """Sixty cycles of one sweep each: the potential grows to nearly twice its
    first value, and once it has outgrown the scale that gives way; the loop of
    launches ends at the same potential."""
    H = I.Hierarchy(dim, [n], [tuple([0.0] * dim)], 1.0 / n, 1.0, [], "const")
    inp = [{"rho": np.ones((n,) * dim), "bc_rho": np.ones((n + 2,) * dim), "bc_phi": np.zeros((n + 4,) * dim)}]
    kw = dict(nu_pre=nu[0], nu_post=nu[1], max_cycles=60, rel_tol=0.0)
    _, a = gpu_solve(mg, H, inp, **kw)
    monkeypatch.setenv("MG_BOTTOM_N64", "8")
    _, b = gpu_solve(mg, H, inp, **kw)
    assert a[0]["cycles"] == b[0]["cycles"] == 60
    assert relmax(a[0]["phi"], b[0]["phi"]) < 1e-12


def _discrete_solution(f, block, h):
    """The discrete problem solved by sine transforms and refined with residuals in long doubles."""
    import scipy.fft as sf
    N, dim, LD = f.shape[0], f.ndim, np.longdouble
    lam = 2.0 * np.cos(np.pi * np.arange(1, N + 1) / (N + 1)) - 2.0
    eig = sum(lam.reshape([-1 if a == q else 1 for q in range(dim)]) for a in range(dim))
    x, c = block.astype(LD), (slice(1, -1),) * dim
    x[c] = 0
    for _ in range(4):
        lap = -2 * dim * x[c]
        for a in range(dim):
            for o in (0, 2):
                lap = lap + x[tuple(slice(o, o + N) if q == a else slice(1, -1) for q in range(dim))]
        r = f.astype(LD) * LD(h) ** 2 - lap
        big = float(np.abs(r).max()) or 1.0
        x[c] += sf.idstn(sf.dstn((r / big).astype(float), type=1) / eig, type=1).astype(LD) * big
    return x


@pytest.mark.parametrize("dim,n", [(3, 8), (3, 16), (3, 31), (2, 23), (2, 64), (2, 158)])
@pytest.mark.parametrize("kind", ["sphere", "random", "constant"])
@pytest.mark.parametrize("nu", [(2, 1), (4, 4)])
def test_fp64_slab_converged_potential_is_unbiased(mg, dim, n, kind, nu):  # noqa: F811
    """The converged potential against the discrete solution.  A right-hand
    side is off by at most half a unit of the level's scale, which is at most
    2^-56 of the largest potential, and half a unit everywhere moves the
    potential by N^2 / 16 (2D 0.0737 N^2 / 2) units at most; as much again and
    eight units are allowed for the sweeps' own rounding.  Floors instead of
    rounding exceed this by ten and more."""
    rng = np.random.default_rng(100 * dim + n)
    h, N = 1.0 / n, n + 2
    if kind == "random":
        phi, rho = rng.standard_normal((n + 4,) * dim), rng.standard_normal((N,) * dim)
    elif kind == "constant":
        phi, rho = np.zeros((n + 4,) * dim), np.ones((N,) * dim)
    else:
        r2 = sum((a - 0.13) ** 2 for a in np.meshgrid(*[(np.arange(n + 4) - 1.5) * h - 0.5] * dim, indexing="ij"))
        phi, rho = -1.0 / np.sqrt(r2 + 0.09), (np.maximum(0.0, 1.0 - r2 / 0.09) ** 3)[(slice(1, -1),) * dim]
    H = I.Hierarchy(dim, [n], [tuple([0.0] * dim)], h, 1.0, [], kind)
    inp = [{"rho": np.ascontiguousarray(rho[(slice(1, -1),) * dim]), "bc_rho": np.ascontiguousarray(rho), "bc_phi": phi}]
    _, g = gpu_solve(mg, H, inp, nu_pre=nu[0], nu_post=nu[1], max_cycles=30, rel_tol=0.0)
    x = _discrete_solution(4.0 * np.pi * rho, phi, h)
    unit = 2.0 ** -56 * float(np.abs(x).max())
    err = float(np.abs(g[0]["phi"] - x[(slice(2, -2),) * dim]).max())
    assert err <= unit * ((1.0 / 8 if dim == 3 else 0.0737) * N ** 2 + 8.0)


@pytest.mark.parametrize("dim,n,prec,solve", [(3, 16, "fp64", True), (2, 64, "fp64", True), (3, 62, "fp64", False),
                                              (3, 30, "mixed", False), (2, 126, "mixed", False)])
@pytest.mark.parametrize("graph", ["1", "0"])
def test_slab_wait_timeout_reports_etimeout(mg, monkeypatch, dim, n, prec, solve, graph):  # noqa: F811
    """With MG_FAULT_SLAB_WAIT=1 one CTA's first wait for its neighbours runs
    out (limit about 1 ms): the launch ends, mg_solve reports MG_ETIMEOUT, the
    handle refuses further work, and a new handle solves as one without the
    fault; for levels that one launch solves and for single V-cycles."""
    import torch
    H, inp = random_single_level(dim, n, 3 * n + dim)
    kw = dict(max_cycles=4, rel_tol=0.0)
    if prec == "mixed":
        kw.update(precision=mg.MG_MIXED, inner_cycles=2)
    monkeypatch.setenv("MG_SOLVE_GRAPH", graph)
    _, before = gpu_solve(mg, H, inp, **kw)
    monkeypatch.setenv("MG_FAULT_SLAB_WAIT", "1")
    h = mg.mg_create_hierarchy([mg.desc_from(H)], mg.options(**kw))
    try:
        dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
        mg.mg_set_density(h, 0, 0, dev(inp[0]["rho"]), dev(inp[0]["bc_rho"]), dev(inp[0]["bc_phi"]))
        with pytest.raises(mg.MGError) as ei:
            mg.mg_solve(h, 1, allow_noconv=True)
        assert ei.value.status == mg.MG_ETIMEOUT, ei.value
        with pytest.raises(mg.MGError) as ei:
            mg.mg_solve(h, 1, allow_noconv=True)
        assert ei.value.status == mg.MG_ESTATE, ei.value
    finally:
        mg.mg_destroy(h)
    monkeypatch.delenv("MG_FAULT_SLAB_WAIT")
    _, after = gpu_solve(mg, H, inp, **kw)
    assert np.array_equal(before[0]["phi"], after[0]["phi"])
