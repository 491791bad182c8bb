"""The one-block tail of a box patch's V-cycle (csrc/mg_box.cu: kx_tail) and
the colour-split phases of the persistent batched solve (csrc/mg_kernels.cu:
split_smooth, split_restrict, split_prolong) at the sizes where their plans
and remainders change."""
import pytest

from paper_2001_02327_gb300 import inputs as I
from tests.test_gpu_box import box_solve, mg, oracle_solve, relmax  # noqa: F401
from tests.test_gpu_parity import _batch_solve

pytestmark = pytest.mark.gpu

# first tail level below its limit and past it, short and long axes (one
# cell per axis at different levels), tie (x_N = 1) and odd sizes, 2D
SHAPES = [(3, (18, 18, 18)), (3, (22, 24, 24)), (3, (26, 28, 26)), (3, (28, 28, 28)), (3, (4, 4, 4)), (3, (100, 4, 6)), (3, (14, 22, 30)), (3, (5, 3, 2)),
          (2, (86, 86)), (2, (90, 88)), (2, (108, 106)), (2, (110, 108)), (2, (300, 2)), (2, (7, 9))]


@pytest.mark.parametrize("dim,n", SHAPES)
@pytest.mark.parametrize("nu", [(2, 1), (0, 2), (3, 0)])
def test_fp64_tail_matches_oracle(mg, dim, n, nu):  # noqa: F811
    """Three V-cycles against the FP64 oracle (the parity bar of the FP64 path)."""
    H = (I.box_3d_sphere if dim == 3 else I.box_2d_disk)(n=n, levels=1)
    inp = I.level_inputs(H)
    _, _, got = box_solve(mg, H, inp, nu_pre=nu[0], nu_post=nu[1], max_cycles=3, rel_tol=0.0)
    ref = oracle_solve(H, inp, nu, 3, 0.0)
    assert relmax(got[0][0], ref[0][0]) < 1e-12


@pytest.mark.parametrize("dim,n", SHAPES + [(3, (34, 34, 34)), (3, (36, 34, 34)), (2, (150, 150)), (2, (156, 154))])
def test_mixed_tail_converges_as_fp64(mg, dim, n):  # noqa: F811
    """FP32 V-cycles through the tail reach the FP64 form's tolerance in its
    cycles, give or take one step, and its solution: a relative residual of
    1e-10 leaves at most 1e-10 times the condition number, below 1e5 here."""
    H = (I.box_3d_sphere if dim == 3 else I.box_2d_disk)(n=n, levels=1)
    inp = I.level_inputs(H)
    kw = dict(nu_pre=2, nu_post=2, max_cycles=60, rel_tol=1e-10)
    _, sa, a = box_solve(mg, H, inp, **kw)
    _, sb, b = box_solve(mg, H, inp, precision=mg.MG_MIXED, inner_max=8, **kw)
    assert sa[0]["status"] == sb[0]["status"] == 0
    assert sb[0]["cycles"] <= sa[0]["cycles"] + 3
    assert relmax(b[0][0], a[0][0]) < 1e-5


@pytest.mark.parametrize("dim,edges", [(3, (9, 10, 11, 12, 15, 17)), (3, (18, 31, 33, 41)), (2, (9, 14, 31, 33, 50))])
def test_persistent_split_phases_equal_graph_branches(mg, monkeypatch, dim, edges):  # noqa: F811
    """Rows whose last vector is partly outside the level, odd fine levels,
    the smallest level above the bottom: cycle counts and potentials of the
    per-phase launches on plain levels."""
    Hs = [(I.config_3d_offset_sphere if dim == 3 else I.config_2d_disk)(n, 1) for n in edges]
    monkeypatch.setenv("MG_SPLIT", "0")
    kw = dict(precision=mg.MG_MIXED, nu_pre=2, nu_post=1, inner_max=8)
    monkeypatch.setenv("MG_PERSIST", "0")
    a = _batch_solve(mg, Hs, True, **kw)
    monkeypatch.setenv("MG_PERSIST", "1")
    b = _batch_solve(mg, Hs, True, **kw)
    for ha, hb in zip(a, b):
        for (pa, Fa, sa), (pb, Fb, sb) in zip(ha, hb):
            assert sa["cycles"] == sb["cycles"] and sb["rel_res"] < 1e-10
            assert relmax(pb, pa) < 1e-10 and relmax(Fb, Fa) < 1e-9
