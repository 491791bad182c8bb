"""GPU checks of the FP64 stencils summed on the integer pipe: the marching
residual and force kernels of large 3D levels (csrc/mg_march.cuh) and the
per-cell sums (csrc/mg_fix.cuh), at sizes off their tiles of 32 x 8 cells, with
fields whose exponents change from plane to plane, and outside the plain range
of exponents."""
import numpy as np
import pytest
import torch

from paper_2001_02327_gb300 import inputs as I
from tests.test_gpu_parity import gpu_solve, mg, omega, random_single_level, relmax  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [94, 95, 97, 127])
def test_large_level_matches_oracle(mg, oracle, n):  # noqa: F811
    """Two FP64 V-cycles on random data: potential and forces at the parity
    bar; the residual norm (sums of n^3 squares in another order) to 1e-12."""
    H, inp = random_single_level(3, n, n)
    _, g = gpu_solve(mg, H, inp, nu_pre=1, nu_post=1, max_cycles=2, rel_tol=0.0)
    ref = oracle.solve_hierarchy(H, inp, 1, 1, 2, 0.0)
    assert relmax(g[0]["phi"], omega(ref[0]["phi"], n, 3)) < 1e-12
    assert relmax(g[0]["F"], ref[0]["F"]) < 1e-12
    assert abs(g[0]["rel_res"] / ref[0]["hist"][-1] - 1) < 1e-11


@pytest.mark.parametrize("n", [30, 96])
@pytest.mark.parametrize("kind", ["growing", "zeros", "tiny", "huge"])
def test_residual_over_changing_exponents(mg, kind, n):  # noqa: F811
    """||b|| and ||r|| of a given start against numpy: fields that grow by
    2^200 through the planes, vanish in half of the box, or lie outside the
    plain exponents (there the FP64 instructions run).  Each cell's residual is
    within 20 roundings of its largest term, so the norms agree to 1e-13."""
    rng = np.random.default_rng(n)
    h = 1.0 / n
    full = rng.standard_normal((n + 4,) * 3)
    if kind == "growing":
        full *= np.exp2(200.0 * np.arange(n + 4) / (n + 3) - 100.0)[:, None, None]
    elif kind == "zeros":
        full[: n // 2] = 0.0
    else:
        full *= 1e-140 if kind == "tiny" else 1e140
    rho = rng.standard_normal((n + 2,) * 3) * np.abs(full).max()
    H = I.Hierarchy(3, [n], [(0.0,) * 3], h, 1.0, [], kind)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    hd = mg.mg_create_hierarchy([mg.desc_from(H)], mg.options(max_cycles=0, rel_tol=1e-10, guess=mg.MG_GUESS_USER))
    try:
        mg.mg_set_density(hd, 0, 0, dev(rho[1:-1, 1:-1, 1:-1]), dev(rho), dev(full))
        mg.mg_set_guess(hd, 0, 0, dev(full[1:-1, 1:-1, 1:-1]))
        _, st = mg.mg_solve(hd, 1, allow_noconv=True)
        F = torch.zeros((3, n, n, n), dtype=torch.float64, device="cuda")
        mg.mg_forces(hd, 0, 0, None, F)
        torch.cuda.synchronize()
        F = F.cpu().numpy()
    finally:
        mg.mg_destroy(hd)
    c = (slice(1, -1),) * 3
    f = 4 * np.pi * rho
    nb = lambda a: (a[:-2, 1:-1, 1:-1] + a[2:, 1:-1, 1:-1] + a[1:-1, :-2, 1:-1] + a[1:-1, 2:, 1:-1]
                    + a[1:-1, 1:-1, :-2] + a[1:-1, 1:-1, 2:])
    ring = full.copy()
    ring[c] = 0.0
    r = f - (nb(full) - 6.0 * full[c]) / h ** 2
    b = f - nb(ring) / h ** 2
    assert abs(st[0][0]["b_norm"] / np.linalg.norm(b) - 1) < 1e-13
    assert abs(st[0][0]["rel_res"] / (np.linalg.norm(r) / np.linalg.norm(b)) - 1) < 1e-13
    for a in range(3):
        ax = 2 - a
        s = lambda o: full[tuple(slice(2 + o, 2 + o + n) if q == ax else slice(2, -2) for q in range(3))]
        ref = -(8.0 * (s(1) - s(-1)) - (s(2) - s(-2))) / (12.0 * h)
        mag = (8.0 * (np.abs(s(1)) + np.abs(s(-1))) + np.abs(s(2)) + np.abs(s(-2))) / (12.0 * h)
        # a block of 32 x 8 cells and up to 129 planes shares one exponent: below
        # 2^-40 of its largest value a cell keeps fewer bits
        big = np.maximum(mag, np.exp2(-40.0) * (np.abs(full).max() if kind == "growing" else 0.0))
        assert np.all(np.abs(F[a] - ref) <= 1e-13 * big)


def test_box_patch_residual_and_forces(mg):  # noqa: F811
    """A box patch of unequal, odd-tiled axes solved to 1e-10: the potential
    satisfies the stencil to the tolerance, the forces are Eq. 2 of it."""
    n = (130, 98, 94)
    H = I.box_3d_sphere(n=n, levels=1)
    inp = I.level_inputs(H)[0]
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    hb = mg.mg_box_create(mg.box_desc_from(H), mg.options(nu_pre=2, nu_post=2, precision=mg.MG_MIXED, inner_max=8))
    try:
        mg.mg_box_set_density(hb, 0, dev(inp["rho"]), dev(inp["bc_rho"]), dev(inp["bc_phi"]))
        _, st = mg.mg_box_solve(hb, 1)
        P = torch.zeros(n[::-1], dtype=torch.float64, device="cuda")
        F = torch.zeros((3,) + n[::-1], dtype=torch.float64, device="cuda")
        mg.mg_box_forces(hb, 0, P, F)
        torch.cuda.synchronize()
        p, F = P.cpu().numpy(), F.cpu().numpy()
    finally:
        mg.mg_box_destroy(hb)
    h = H.h(0)
    lap = (p[:-2, 1:-1, 1:-1] + p[2:, 1:-1, 1:-1] + p[1:-1, :-2, 1:-1] + p[1:-1, 2:, 1:-1] + p[1:-1, 1:-1, :-2]
           + p[1:-1, 1:-1, 2:] - 6.0 * p[1:-1, 1:-1, 1:-1]) / h ** 2
    r = 4 * np.pi * inp["rho"][1:-1, 1:-1, 1:-1] - lap
    assert st[0]["rel_res"] < 1e-10 and np.linalg.norm(r) <= 1.001 * st[0]["rel_res"] * st[0]["b_norm"]
    i = (slice(2, -2),) * 3
    for a in range(3):
        ax = 2 - a
        s = lambda o: p[tuple(slice(2 + o, p.shape[q] - 2 + o) if q == ax else slice(2, -2) for q in range(3))]
        ref = -(8.0 * (s(1) - s(-1)) - (s(2) - s(-2))) / (12.0 * h)
        assert np.max(np.abs(F[a][i] - ref)) <= 1e-13 * np.max(np.abs(p)) / h


def _differences(full, ax, n, stencil):
    """Numerator of the force difference along array axis ax over the inner n cells per axis, and the sum of
    the magnitudes of the differences that it is made of, in long doubles."""
    v = full.astype(np.longdouble)
    s = lambda o: v[tuple(slice(2 + o, 2 + o + m) if q == ax else slice(2, 2 + k)
                          for q, (m, k) in enumerate(zip(n, n)))]
    if stencil == 1:
        d = s(1) - s(-1)
        return d, np.abs(d)
    d1, d2 = s(1) - s(-1), s(2) - s(-2)
    return 8 * d1 - d2, 8 * np.abs(d1) + np.abs(d2)


@pytest.mark.parametrize("n", [30, 95, 96, 131])
@pytest.mark.parametrize("kind", ["growing", "steep", "smooth", "plateau"])
@pytest.mark.parametrize("stencil", [0, 1])
def test_forces_no_less_accurate_than_fp64(mg, kind, n, stencil):  # noqa: F811
    """Every cell's force within the rounding of the FP64 expression: one 2^-53
    of each difference, of their difference, of the factor (two) and of the
    product, 6 x 2^-53 of the sum of the differences' magnitudes.  Fields that
    grow by 2^200 and by 2^12 per 32 cells, a smooth one, and one that is large
    in a few planes and smooth far below them."""
    rng = np.random.default_rng(n)
    h = 1.0 / n
    z, y, x = np.meshgrid(*[np.arange(n + 4, dtype=float)] * 3, indexing="ij")
    full = 1.0 / np.sqrt((x - 0.3 * n) ** 2 + (y - 0.6 * n) ** 2 + (z - 0.5 * n) ** 2 + 9.0)
    if kind == "growing":
        full = rng.standard_normal(full.shape) * np.exp2(200.0 * z / (n + 3) - 100.0)
    elif kind == "steep":
        full *= np.exp2((x + z) * (12.0 / 32.0))
    elif kind == "plateau":
        full *= np.where((z.astype(int) % 40) < 3, 1000.0, 1.0)
    H = I.Hierarchy(3, [n], [(0.0,) * 3], h, 1.0, [], kind)
    rho = rng.standard_normal((n + 2,) * 3)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    hd = mg.mg_create_hierarchy([mg.desc_from(H)], mg.options(max_cycles=0, guess=mg.MG_GUESS_USER, force_stencil=stencil))
    try:
        mg.mg_set_density(hd, 0, 0, dev(rho[1:-1, 1:-1, 1:-1]), dev(rho), dev(full))
        mg.mg_set_guess(hd, 0, 0, dev(full[1:-1, 1:-1, 1:-1]))
        mg.mg_solve(hd, 1, allow_noconv=True)
        F = torch.zeros((3, n, n, n), dtype=torch.float64, device="cuda")
        mg.mg_forces(hd, 0, 0, None, F)
        torch.cuda.synchronize()
        F = F.cpu().numpy()
    finally:
        mg.mg_destroy(hd)
    c = (12 if stencil == 0 else 2) * np.longdouble(h)
    for a in range(3):
        s, mag = _differences(full, 2 - a, (n,) * 3, stencil)
        assert np.all(np.abs(F[a] + s / c) <= 6 * 2.0 ** -53 * mag / c)


def test_box_forces_no_less_accurate_than_fp64(mg):  # noqa: F811
    """The same for a box patch that the marching kernel takes, of its solved potential."""
    n = (130, 98, 94)
    H = I.box_3d_sphere(n=n, levels=1)
    inp = I.level_inputs(H)[0]
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    hb = mg.mg_box_create(mg.box_desc_from(H), mg.options(nu_pre=2, nu_post=2, precision=mg.MG_MIXED, inner_max=8))
    try:
        mg.mg_box_set_density(hb, 0, dev(inp["rho"]), dev(inp["bc_rho"]), dev(inp["bc_phi"]))
        mg.mg_box_solve(hb, 1)
        P = torch.zeros(n[::-1], dtype=torch.float64, device="cuda")
        F = torch.zeros((3,) + n[::-1], dtype=torch.float64, device="cuda")
        mg.mg_box_forces(hb, 0, P, F)
        torch.cuda.synchronize()
        p, F = P.cpu().numpy(), F.cpu().numpy()
    finally:
        mg.mg_box_destroy(hb)
    i, c = (slice(2, -2),) * 3, 12 * np.longdouble(H.h(0))
    for a in range(3):
        s, mag = _differences(p, 2 - a, tuple(m - 4 for m in p.shape), 0)
        assert np.all(np.abs(F[a][i] + s / c) <= 6 * 2.0 ** -53 * mag / c)
