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
