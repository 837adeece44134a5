"""The solver's kernels at the sizes where their partitions end: camera counts around the update
kernels' 14 cameras per CTA and the Gram kernel's 64 rows, direction widths 1 to 16, histories past the
reorthogonalisation's tiles, and residuals far from one (the float32 sweeps solve for the residual
divided by a power of two), and the camera counts up to which one CTA (float32 sweeps, 20) or one
cluster (float64 PCG, 24) solves a problem."""
import numpy as np
import pytest

from oracle import lm as olm
from oracle import solvers as osol
from paper_2110_04015_gb300 import binding, problem
from paper_2110_04015_gb300 import synthetic as sy
from tests._gpu import energy_err

pytestmark = pytest.mark.gpu


def _system(n_cams, n_pts, **kw):
    sc = sy.tiny(n_cams, n_cams=n_cams, n_pts=n_pts, track_min=min(3, n_cams), track_max=min(6, n_cams), **kw)
    m = olm.measurements(sc)
    return sc, m, olm.linearise(sc.cams0, sc.pts0, sc.obs_cam, sc.obs_pt, m, 1e-4)


SOLVES = (None, (8, 3.0), (16, 1e9), (3, 0.0), (11, 6.0), (5, 1e9))


def _solve(p, args, tol):
    return p.ba_solve_pcg(tol, 5000) if args is None else p.ba_solve_mcg(tol, 5000, *args)


# The stop test is on the residual |-b~ - S x| <= tol |b~|, so that is what is checked (float64: the
# recursive residual stops, and the true one stays within 1.5 of it), together with the energy norm of
# the error against the dense solution, at the bound that the other tests hold solves to 1e-6 to.
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("n_cams", [2, 3, 7, 8, 14, 15, 20, 21, 24, 25, 28, 43, 57])
def test_camera_counts_around_the_partitions(n_cams, precision):
    sc, m, lin = _system(n_cams, 45 * n_cams + 7)
    ref = osol.dense_solve(lin.S, lin.btilde)
    with binding.Problem(sc.cams0, sc.pts0, sc.obs_cam, sc.obs_pt, m, precision=precision) as p:
        p.ba_build_normal(1e-4)
        for args in SOLVES:
            st = _solve(p, args, 1e-11)
            assert st["status"] == 0, (args, st)
            assert st["true_rel_residual"] <= (1e-11 if precision == "mixed" else 1.5e-11), (args, st)
            assert energy_err(lin.S, p.ba_get_delta().ravel(), ref) < 1e-4, args


# Measurements that the starting point already fits to rel of a parameter: b~ shrinks with rel, and the
# third float32 sweep starts 1e12 below it.
@pytest.mark.parametrize("rel", [1e-3, 1e-6, 1e-9])
def test_sweeps_on_small_residuals_converge(rel):
    sc, m, _ = _system(16, 1000, sigma=0.0, rel_perturb=rel)
    with binding.Problem(sc.cams0, sc.pts0, sc.obs_cam, sc.obs_pt, m, precision="mixed") as p:
        p.ba_build_normal(1e-4)
        for args in SOLVES[:3]:
            st = _solve(p, args, 1e-12)
            assert st["status"] == 0 and st["true_rel_residual"] <= 1e-12, (args, st)


# Problems on both sides of those counts in one batch: each gives the bits of its solo solve.
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_small_problems_in_a_batch_give_their_solo_bits(precision):
    scenes = [sy.tiny(n, n_cams=n, n_pts=50 * n) for n in (13, 30, 20, 24, 60, 21, 7)]
    solo = []
    for sc in scenes:
        with problem.from_scene(sc, precision=precision) as p:
            p.ba_build_normal(1e-4)
            solo.append([(_solve(p, a, 1e-9), p.ba_get_delta().copy())[1] for a in SOLVES])
    off = np.cumsum([0] + [sc.n_cams for sc in scenes])
    with problem.from_scenes(scenes, precision=precision) as b:
        b.ba_build_normal(1e-4)
        for k, a in enumerate(SOLVES):
            assert _solve(b, a, 1e-9)["status"] == 0
            x = b.ba_get_delta()
            for q in range(len(scenes)):
                assert np.array_equal(x[off[q]:off[q + 1]], solo[q][k]), (a, scenes[q].n_cams)


# Direction counts on both sides of 8, up to which two lanes share a block in the multi-column product,
# on problems that run it (more than 20 cameras), every step local.
@pytest.mark.parametrize("dirs", [2, 4, 7, 8, 9, 16])
def test_local_steps_of_every_width_class(dirs):
    sc, m, lin = _system(45, 1500)
    ref = osol.dense_solve(lin.S, lin.btilde)
    with binding.Problem(sc.cams0, sc.pts0, sc.obs_cam, sc.obs_pt, m, precision="mixed") as p:
        p.ba_build_normal(1e-4)
        st = p.ba_solve_mcg(1e-11, 5000, dirs, 1e9)
        assert st["status"] == 0 and st["local_steps"] > 0 and st["true_rel_residual"] <= 1e-11, st
        assert energy_err(lin.S, p.ba_get_delta().ravel(), ref) < 1e-4


# The same scene in other length units: translations and landmarks times s give the same residuals, and a
# scaled system (Lam S Lam) that differs only through the damping's floor, while Lam and the unscaled
# residual change by factors of s and 1 / s.  A float32 sweep must not depend on them: 16 cameras run in one
# CTA, 45 in the kernels of an iteration.
@pytest.mark.parametrize("n_cams", [16, 45])
@pytest.mark.parametrize("s", [1e-12, 1e-9, 1e-6, 1e6])
def test_length_units_do_not_leave_the_float32_range(n_cams, s):
    sc, m, _ = _system(n_cams, 60 * n_cams)
    cams = sc.cams0.copy()
    cams[:, 3:6] *= s
    with binding.Problem(cams, sc.pts0 * s, sc.obs_cam, sc.obs_pt, m, precision="mixed") as p:
        p.ba_build_normal(1e-4)
        for args in SOLVES:
            st = _solve(p, args, 1e-10)
            assert st["status"] == 0 and st["true_rel_residual"] <= 1e-10, (args, st)


# Residuals far from one in the kernels of an iteration (problems of up to 20 cameras run in one CTA).  The
# true residual in double-float is good to 2^-48 |S| |x|, at most about 1e3 |b~| 2^-48 = 4e-12 |b~| here.
@pytest.mark.parametrize("rel", [1e-3, 1e-6, 1e-9])
def test_sweeps_on_small_residuals_converge_above_one_cta(rel):
    sc, m, _ = _system(45, 2700, sigma=0.0, rel_perturb=rel)
    with binding.Problem(sc.cams0, sc.pts0, sc.obs_cam, sc.obs_pt, m, precision="mixed") as p:
        p.ba_build_normal(1e-4)
        for args in SOLVES[:3]:
            st = _solve(p, args, 1e-11)
            assert st["status"] == 0 and st["true_rel_residual"] <= 1e-11, (args, st)


# A problem that one CTA solves waits for no tile, so its solve launches no tile-streaming product: a sweep by MCG
# is as many launches as one by PCG (its start, the one CTA, the loop test, the true residual and the next
# sweep's plan), after the three launches that start the refinement.
def test_one_cta_solves_launch_no_product():
    sc, m, _ = _system(13, 777)
    with binding.Problem(sc.cams0, sc.pts0, sc.obs_cam, sc.obs_pt, m, precision="mixed") as p:
        p.ba_build_normal(1e-4)
        per_sweep = []
        for args in (None, (8, 3.0), (4, 1e9)):
            before = p.ba_get_launch_count()
            sweeps = _solve(p, args, 1e-6)["refinements"]
            per_sweep.append((p.ba_get_launch_count() - before - 3) / sweeps)
        assert per_sweep[0] == per_sweep[1] == per_sweep[2], per_sweep


# Direction counts on both sides of 10, up to which one CTA runs MCG on up to 20 cameras (16 cameras: subsets of
# one and two cameras), every step local and none, alone and beside problems that the other path takes.
@pytest.mark.parametrize("dirs", [2, 5, 8, 10, 11, 15, 16])
def test_direction_counts_around_the_one_cta_limit(dirs):
    scenes = [sy.tiny(n, n_cams=n, n_pts=60 * n) for n in (10, 11, 16, 20, 30)]
    solo = []
    for sc in scenes:
        with problem.from_scene(sc, precision="mixed") as p:
            p.ba_build_normal(1e-4)
            for tau in (1e9, 0.0):
                st = p.ba_solve_mcg(1e-9, 5000, dirs, tau)
                assert st["status"] == 0 and st["true_rel_residual"] <= 1e-9, (sc.n_cams, tau, st)
                solo.append(p.ba_get_delta().copy())
    off = np.cumsum([0] + [sc.n_cams for sc in scenes])
    with problem.from_scenes(scenes, precision="mixed") as b:
        b.ba_build_normal(1e-4)
        for k, tau in enumerate((1e9, 0.0)):
            assert b.ba_solve_mcg(1e-9, 5000, dirs, tau)["status"] == 0
            x = b.ba_get_delta()
            for q in range(len(scenes)):
                assert np.array_equal(x[off[q]:off[q + 1]], solo[2 * q + k]), (tau, scenes[q].n_cams)


# A full history ends a float32 sweep; one CTA keeps its history in tiles of 64 columns, so capacities around them.
@pytest.mark.parametrize("cap", [9, 40, 63, 64, 65, 130])
def test_full_histories_of_one_cta_sweeps(cap):
    sc, m, _ = _system(13, 777)
    with binding.Problem(sc.cams0, sc.pts0, sc.obs_cam, sc.obs_pt, m, precision="mixed", max_history=cap,
                         max_refine=2000) as p:
        p.ba_build_normal(1e-2)
        for args in ((8, 3.0), (4, 1e9), (10, 0.0)):
            st = p.ba_solve_mcg(1e-8, 20000, *args)
            assert st["status"] == 0 and st["true_rel_residual"] <= 1e-8 and st["history_cols"] <= cap, (args, st)


# Batches of more than 19 problems run small CTAs where fewer problems have large ones and clusters: the same bits
# as alone.  With a problem of 230 cameras in it the small solves keep their clusters.
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("largest", [70, 230])
def test_many_problems_give_their_solo_bits(precision, largest):
    sizes = [9, 16, 21, 30, 45, largest]
    scenes = [sy.tiny(n, n_cams=n, n_pts=40 * n) for n in sizes]
    solves = ((3, 3.0), (8, 1e9), (16, 10.0), (5, 0.0))
    solo = []
    for sc in scenes:
        with problem.from_scene(sc, precision=precision) as p:
            p.ba_build_normal(1e-3)
            solo.append([(p.ba_solve_mcg(1e-6, 2000, *a), p.ba_get_delta().copy())[1] for a in solves])
    batch = scenes * 4   # 24 problems
    off = np.cumsum([0] + [sc.n_cams for sc in batch])
    with problem.from_scenes(batch, precision=precision) as b:
        b.ba_build_normal(1e-3)
        for k, a in enumerate(solves):
            assert b.ba_solve_mcg(1e-6, 2000, *a)["status"] == 0
            x = b.ba_get_delta()
            for q in range(len(batch)):
                assert np.array_equal(x[off[q]:off[q + 1]], solo[q % len(scenes)][k]), (a, batch[q].n_cams, q)


# Handles of more than 3600 cameras form the preconditioner with a thread per camera instead of a warp: the same bits
# as each problem alone, on both sides of the limit and with a last CTA that is not full.
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("problems", [225, 226, 229])
def test_preconditioner_of_many_cameras_gives_the_solo_bits(precision, problems):
    scenes = [sy.tiny(i, n_cams=16, n_pts=200) for i in range(3)]
    solo = []
    for sc in scenes:
        with problem.from_scene(sc, precision=precision) as p:
            p.ba_build_normal(1e-3)
            p.ba_solve_pcg(1e-6, 1000)
            solo.append((p.ba_get_preconditioner().copy(), p.ba_get_delta().copy()))
    with problem.from_scenes([scenes[b % 3] for b in range(problems)], precision=precision) as b:
        b.ba_build_normal(1e-3)
        b.ba_solve_pcg(1e-6, 1000)
        D, x = b.ba_get_preconditioner(), b.ba_get_delta()
        for q in range(problems):
            assert np.array_equal(D[16 * q:16 * q + 16], solo[q % 3][0]), q
            assert np.array_equal(x[16 * q:16 * q + 16], solo[q % 3][1]), q


# spmv_config 1 means 8 warps x 1 stage in float64, today's default shape too: the same product in the same time
# (the other shapes take 1.4 and 2.8 times as long here).
def test_float64_shape_1_is_8_warps():
    sc = sy.dense(1, n_cams=1000, n_pts=100000, n_clusters=33)
    xy = problem.device_measurements(sc)
    ms, x = [], []
    for cfg in (0, 1):
        with problem.from_scene(sc, xy=xy, spmv_config=cfg) as p:
            p.ba_build_normal(1e-4)
            p.ba_time_kernel("spmv", 5)
            ms.append(min(p.ba_time_kernel("spmv", 10) for _ in range(3)))
            p.ba_solve_pcg(1e-6, 1000)
            x.append(p.ba_get_delta().copy())
    assert ms[1] < 1.2 * ms[0], ms
    assert np.array_equal(x[0], x[1])


# The network's centre features are standardised per axis, so a power of two as the length unit changes no bit of them,
# however far the squares of the coordinates are from float32's range.
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("k", [-70, -20, 20, 62])
def test_network_features_do_not_depend_on_the_length_unit(k, precision):
    sc, m, _ = _system(24, 1200)
    X = []
    for s in (1.0, 2.0 ** k):
        cams = sc.cams0.copy()
        cams[:, 3:6] *= s
        with binding.Problem(cams, sc.pts0 * s, sc.obs_cam, sc.obs_pt, m, precision=precision) as p:
            if k == -70 and precision == "mixed" and s < 1.0:   # the float32 build has no such range
                with pytest.raises(binding.BAError) as e:
                    p.ba_build_normal(1e-4)
                assert e.value.code == binding.BA_ERR_SINGULAR
                return
            p.ba_build_normal(1e-4)
            g = binding.GNN(np.zeros(17537, np.float32))
            X.append(g.ba_gnn_graph(p)[0])
            g.close()
    assert np.array_equal(X[0][:, :6], X[1][:, :6])


# In a batch with larger problems the small ones run beside their iterations, not before them: the batch takes less than
# the larger problems and the small ones one after the other (measured 9.9 against 8.9 + 2.6 ms).
def test_small_problems_run_beside_larger_ones():
    small = [sy.tiny(i, n_cams=20, n_pts=1500) for i in range(8)]
    large = [sy.dense(i, n_cams=300, n_pts=30000, n_clusters=10) for i in range(8)]
    ms = []
    for scenes in (small, large, small + large):
        with problem.from_scenes(scenes, precision="mixed") as b:
            b.ba_build_normal(1e-4)
            t = [b.ba_solve_mcg(1e-9, 1000, 8, 3.0)["ms"] for _ in range(7)]
            ms.append(float(np.median(t)))
    assert ms[2] < ms[1] + 0.75 * ms[0], ms
