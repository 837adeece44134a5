"""The solver's kernels at the sizes where their partitions end: camera counts around the update
kernels' 14 cameras per CTA, histories around the reorthogonalisation's tiles, and residuals far from
one (the float32 sweeps solve for the residual divided by a power of two)."""
import numpy as np
import pytest

from oracle import lm as olm
from oracle import solvers as osol
from paper_2110_04015_gb300 import binding
from paper_2110_04015_gb300 import synthetic as sy

pytestmark = pytest.mark.gpu


def _system(n_cams, n_pts, **kw):
    sc = sy.tiny(n_cams, n_cams=n_cams, n_pts=n_pts, track_min=min(3, n_cams), track_max=min(6, n_cams), **kw)
    m = olm.measurements(sc)
    lin = olm.linearise(sc.cams0, sc.pts0, sc.obs_cam, sc.obs_pt, m, 1e-4)
    return sc, m, osol.dense_solve(lin.S, lin.btilde).reshape(n_cams, 9)


def _solve_all(sc, m, ref, precision, tol, bound):
    scale = np.abs(ref).max(axis=0)
    with binding.Problem(sc.cams0, sc.pts0, sc.obs_cam, sc.obs_pt, m, precision=precision) as p:
        p.ba_build_normal(1e-4)
        for args in (None, (8, 3.0), (16, 1e9), (3, 0.0)):
            st = p.ba_solve_pcg(tol, 5000) if args is None else p.ba_solve_mcg(tol, 5000, *args)
            assert st["status"] == 0, (args, st)
            if precision == "mixed":
                assert st["true_rel_residual"] <= tol, (args, st)
            err = float((np.abs(p.ba_get_delta() - ref) / scale).max())
            assert err < bound, (args, err)


# The reduced systems of these scenes have scaled condition numbers up to about 1e4, so a relative
# residual of 1e-11 leaves at most 1e-7 of each parameter's largest update.
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("n_cams", [2, 3, 14, 15, 28, 43, 57])
def test_camera_counts_around_the_update_chunks(n_cams, precision):
    sc, m, ref = _system(n_cams, 45 * n_cams + 7)
    _solve_all(sc, m, ref, precision, 1e-11, 1e-7)


# Measurements that the starting point already fits to rel of a parameter: b~ shrinks with rel, and the
# third float32 sweep starts 1e12 below it.  The solver's own contract is checked (its double-float true
# residual): the update itself is then only as good as the residuals pi - m, which cancel.
@pytest.mark.parametrize("rel", [1e-3, 1e-6, 1e-9])
def test_sweeps_on_small_residuals_converge(rel):
    sc, m, _ = _system(16, 1000, sigma=0.0, rel_perturb=rel)
    with binding.Problem(sc.cams0, sc.pts0, sc.obs_cam, sc.obs_pt, m, precision="mixed") as p:
        p.ba_build_normal(1e-4)
        for args in (None, (8, 3.0), (16, 1e9)):
            st = p.ba_solve_pcg(1e-12, 5000) if args is None else p.ba_solve_mcg(1e-12, 5000, *args)
            assert st["status"] == 0 and st["true_rel_residual"] <= 1e-12, (args, st)
