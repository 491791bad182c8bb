"""What a handle costs before its second solve."""
import time

import numpy as np
import pytest

from paper_2001_02327_gb300 import inputs as I
from tests.test_gpu_parity import mg  # noqa: F401

pytestmark = pytest.mark.gpu


def _batch(mg, edges, count, **kw):  # noqa: F811
    import torch
    Hs = [I.config_3d_offset_sphere(edges[b % len(edges)], 2) for b in range(count)]
    inp = {H.n[0]: [{k: torch.from_numpy(np.ascontiguousarray(v)).cuda() for k, v in lev.items()}
                    for lev in I.level_inputs(H)] for H in Hs[:len(edges)]}
    h = mg.mg_create_hierarchy([mg.desc_from(H) for H in Hs], mg.options(**kw))
    for b, H in enumerate(Hs):
        for l, lev in enumerate(inp[H.n[0]]):
            mg.mg_set_density(h, b, l, *([lev["rho"], lev["bc_rho"], lev["bc_phi"]] if l == 0 else [lev["rho"]]))
    torch.cuda.synchronize()
    return h


def _solve_ms(mg, h, count):  # noqa: F811
    t = time.perf_counter()
    mg.mg_solve(h, count)
    return 1e3 * (time.perf_counter() - t)


def test_first_solve_of_a_persistent_batch_costs_little_more_than_the_next(mg):  # noqa: F811
    """The plan of the persistent launch changes the storage layout of every
    level, whose arrays are zero until something runs on them: nothing to
    clear.  Building and instantiating a graph of one kernel and copying the
    plan take well under the solve's own time; one memset per array took more
    than twice that time."""
    count, first, later = 256, [], []
    for _ in range(3):
        h = _batch(mg, (16, 24, 32), count, precision=mg.MG_MIXED, nu_pre=2, nu_post=1, inner_max=8)
        try:
            first.append(_solve_ms(mg, h, count))
            assert mg.mg_persistent_count(h) == count
            later.append(min(_solve_ms(mg, h, count) for _ in range(2)))
        finally:
            mg.mg_destroy(h)
    assert min(first) < 2.0 * min(later)


def test_layout_change_after_a_solve_clears_the_arrays(mg, monkeypatch):  # noqa: F811
    """A batch solved by graph branches, then, on the same handle, by the
    persistent launch (another layout of the FP32 arrays), and back: potentials
    of handles that only ever ran one form."""
    import torch
    count = 6
    kw = dict(precision=mg.MG_MIXED, nu_pre=2, nu_post=1, inner_max=8)

    def phis(h):
        out = []
        for b in range(count):
            n = (16, 28, 36)[b % 3]
            p = torch.zeros((n,) * 3, dtype=torch.float64, device="cuda")
            mg.mg_forces(h, b, 1, p, None)
            torch.cuda.synchronize()
            out.append(p.cpu().numpy())
        return out

    want = {}
    for mode in ("0", "1"):
        monkeypatch.setenv("MG_PERSIST", mode)
        h = _batch(mg, (16, 28, 36), count, **kw)
        mg.mg_solve(h, count)
        want[mode] = phis(h)
        mg.mg_destroy(h)
    h = _batch(mg, (16, 28, 36), count, **kw)
    outputs = [torch.zeros((4,) + (16,) * 3, dtype=torch.float64, device="cuda") for _ in range(4)]
    try:
        for out, mode in zip(outputs, ("0", "1", "0", "1")):
            monkeypatch.setenv("MG_PERSIST", mode)
            mg.mg_set_outputs(h, 0, 0, out[0], out[1:])   # another output array: the solve graph is built anew
            mg.mg_solve(h, count)
            for a, b in zip(phis(h), want[mode]):
                assert np.max(np.abs(a - b)) <= 1e-10 * np.max(np.abs(b))
    finally:
        mg.mg_destroy(h)


def test_creation_with_the_slab_kernel_costs_little_more_than_without(mg, monkeypatch):  # noqa: F811
    """Three levels of three sizes: the slab kernel's plans (a matrix of 64
    columns on the host, a launch and a copy per size, no allocation, no wait)
    in place of the one-block kernel's (a launch and a wait per level).  With an
    allocation and two waits per size, and both plans, it took twice the time."""
    H = I.Hierarchy(3, [30, 28, 26], [(-0.5,) * 3, (-0.5 + 8 / 30,) * 3, (-0.5 + 12 / 30,) * 3], 1.0 / 30, 1.0, [], "abc")

    def create_ms(env):
        if env:
            monkeypatch.setenv("MG_BOTTOM_N64", "8")
        else:
            monkeypatch.delenv("MG_BOTTOM_N64", raising=False)
        t0 = time.perf_counter()
        h = mg.mg_create_hierarchy([mg.desc_from(H)], mg.options())
        t = 1e3 * (time.perf_counter() - t0)
        mg.mg_destroy(h)
        return t

    pairs = [(create_ms(True), create_ms(False)) for _ in range(30)]   # in turn, the quickest of each
    assert min(b for _, b in pairs) < 1.5 * min(a for a, _ in pairs)
