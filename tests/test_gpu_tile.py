"""Element-tile sweep against the FP64 oracle at the sizes where its layout
can go wrong: one-element subdomains, several subdomains per warp (with a
last warp that is not full), idle lanes and bands, chains of their own warps,
clusters with slabs of unequal height, both tile shapes, a source, the
WaveHoltz tolerance, rank-local rectangles, non-square elements.

The same for the one-element-per-thread kernel on curved quadrilaterals.

Bounds: FP64 1e-12 and FP32 fp32_bound (the bounds of the other kernels: the
tiles sum the same terms in another order); the tolerance mode may stop one
iteration apart near the threshold, so it is bounded by 10 x the tolerance.
"""

import numpy as np
import pytest

import _tolerances as _tol
from test_gpu_parity import _dev, _host_c, _pair, _rand_lam, _rel, _run_sweep, _wl

pytestmark = pytest.mark.gpu

LAYOUTS = [  # nx, ny, sub_nx, sub_ny, P
    (3, 3, 1, 1, 2),      # one element: chains of one element, 16 subdomains per warp
    (6, 4, 2, 2, 5),      # 6 subdomains, 8 per warp
    (12, 4, 4, 4, 3),     # 3 subdomains, 2 (one element per tile) or 4 (two) per warp
    (16, 16, 8, 8, 3),    # the benchmark's subdomain: one warp in the paired shape
    (16, 8, 8, 8, 1),
    (10, 12, 5, 6, 2),    # idle lanes (5 of 8) and bands
    (7, 9, 7, 3, 4),      # odd element rows
    (17, 4, 17, 2, 3),    # 17 of 32 lanes, chain B longer than the tile rows
    (24, 22, 12, 22, 3),  # a cluster of slabs of unequal height
    (16, 32, 16, 32, 5),  # P = 5, several slabs
    (64, 32, 32, 32, 4),  # the 1024^2 workload's subdomain
]


def _force(monkeypatch, shape):
    monkeypatch.setenv("HZ_SWEEP_VARIANT", "tile")
    monkeypatch.setenv("HZ_TILE_SHAPE", str(shape))


@pytest.mark.parametrize("shape", [1, 2])
@pytest.mark.parametrize("nx,ny,sx,sy,P", LAYOUTS)
def test_tile_sweep_fp32_matches_oracle(hz, monkeypatch, nx, ny, sx, sy, P, shape):
    if shape == 2 and (sy % 2 or P > 3):
        pytest.skip("paired tiles need an even number of element rows and P <= 3")
    _force(monkeypatch, shape)
    case, pr = _pair(hz, _wl(nx, ny, sx, sy, P, box=(0.0, 1.0, 0.0, 0.7)), g_seed=nx + P)
    nt = hz.hz_problem_nt(case.pr)
    lam = _rand_lam(pr, 5)
    bound = _tol.fp32_bound(sx * P + 1)
    for with_rhs in (True, False):
        got_l, got_u = _run_sweep(hz, case, pr, hz.HZ_FP32_REFINE, nt, 4, lam, with_rhs)
        ref_l, ref_u, _ = pr.sweep(lam, pr.rhs() if with_rhs else None, nt, 4, want_u=True)
        assert _rel(got_u, ref_u) < bound and _rel(got_l, ref_l) < bound, with_rhs
    _, u = _run_sweep(hz, case, pr, hz.HZ_FP32_REFINE, nt, 30, lam, False, wh_tol=1e-3)
    _, ref_u, _ = pr.sweep(lam, None, nt, 30, wh_tol=1e-3, want_u=True)
    assert _rel(u, ref_u) < 1e-2
    case.close()


@pytest.mark.parametrize("nx,ny,sx,sy,P", [v for v in LAYOUTS if v[4] <= 4])
def test_tile_sweep_fp64_matches_oracle(hz, monkeypatch, nx, ny, sx, sy, P):
    _force(monkeypatch, 1)
    case, pr = _pair(hz, _wl(nx, ny, sx, sy, P, box=(0.0, 1.0, 0.0, 0.7)), g_seed=nx + P)
    nt = hz.hz_problem_nt(case.pr)
    lam = _rand_lam(pr, 6)
    for with_rhs in (True, False):
        got_l, got_u = _run_sweep(hz, case, pr, hz.HZ_FP64, nt, 2, lam, with_rhs)
        ref_l, ref_u, _ = pr.sweep(lam, pr.rhs() if with_rhs else None, nt, 2, want_u=True)
        assert _rel(got_u, ref_u) < 1e-12 and _rel(got_l, ref_l) < 1e-12, with_rhs
    case.close()


@pytest.mark.parametrize("sx,sy,P,shape", [(4, 4, 2, 1), (8, 8, 3, 2), (32, 32, 4, 1)])
def test_tile_rectangles_equal_the_whole_sweep_bitwise(hz, monkeypatch, sx, sy, P, shape):
    """Rank-local sweeps of two rectangles write what one sweep writes, bit for bit."""
    import torch

    _force(monkeypatch, shape)
    case, pr = _pair(hz, _wl(3 * sx, 2 * sy, sx, sy, P))
    nt, lam = hz.hz_problem_nt(case.pr), _rand_lam(pr, 7)
    whole_l, whole_u = _run_sweep(hz, case, pr, hz.HZ_FP32_REFINE, nt, 2, lam, False)
    lin, lout = _dev(lam), torch.zeros(2 * lam.size, dtype=torch.float64, device="cuda")
    u = torch.zeros(2 * whole_u.size, dtype=torch.float64, device="cuda")
    for rect in ((0, 0, 1, 2), (1, 0, 2, 2)):
        hz.hz_sweep_rect(case.pr, hz.HZ_FP32_REFINE, nt, 2, 0.0, rect, lin, lout, None, u)
    torch.cuda.synchronize()
    assert np.array_equal(_host_c(u).reshape(whole_u.shape), whole_u)
    assert np.array_equal(_host_c(lout).reshape(whole_l.shape), whole_l)
    case.close()


@pytest.mark.parametrize("nx,ny,sx,sy,P", [
    (3, 3, 1, 1, 2),      # one element, 32 subdomains per warp
    (12, 4, 4, 4, 3),     # 3 subdomains, 2 per warp
    (16, 16, 8, 8, 3),    # the curved benchmark's subdomain: 2 warps
    (10, 12, 5, 6, 4),    # idle lanes
    (34, 6, 17, 3, 1),    # 17 of 32 lanes
])
def test_curved_tile_sweep_matches_oracle(hz, monkeypatch, nx, ny, sx, sy, P):
    from paper_2606_21695_gb300.api import Case
    from oracle import geom, sem
    from workloads import configs

    monkeypatch.setenv("HZ_SWEEP_VARIANT", "tile")
    for robin in ((0.0, 1.0), (0.3, 0.8)):
        wl = configs.Workload("ct", (0.0, 1.0, 0.0, 0.8), nx, ny, P, sx, sy, 9.0, "channel", (0.37, 0.48), 0.08,
                              extra={"warp": 0.04})
        case = Case(wl)
        hz.hz_problem_set(case.pr, hz.HZ_TRANSMISSION, np.array(robin))
        m = sem.Mesh(*wl.box, nx, ny, P, sx, sy)
        X, Y = wl.node_xy(*m.coords_1d())
        pr = geom.MappedProblem(m, X, Y, wl.speed_at(X, Y), wl.omega, wl.source_at(X, Y), wl.boundary(), robin=robin)
        nt, lam = hz.hz_problem_nt(case.pr), _rand_lam(pr, 8)
        for with_rhs in (True, False):
            got_l, got_u = _run_sweep(hz, case, pr, hz.HZ_FP32_REFINE, nt, 3, lam, with_rhs)
            ref_l, ref_u, _ = pr.sweep(lam, pr.rhs() if with_rhs else None, nt, 3, want_u=True)
            assert _rel(got_u, ref_u) < _tol.FP32_REL and _rel(got_l, ref_l) < _tol.FP32_REL, (robin, with_rhs)
        _, u = _run_sweep(hz, case, pr, hz.HZ_FP32_REFINE, nt, 30, lam, False, wh_tol=1e-3)
        _, ref_u, _ = pr.sweep(lam, None, nt, 30, wh_tol=1e-3, want_u=True)
        assert _rel(u, ref_u) < 1e-2
        case.close()


@pytest.mark.parametrize("nx,ny,sx,sy,P,shape,precision", [
    (24, 22, 12, 22, 3, 1, "fp32"),   # two slabs: the two that wait for each other
    (64, 32, 32, 32, 3, 2, "fp32"),
    (64, 32, 32, 32, 4, 1, "fp32"),   # more than two: slabs that saw nothing amiss themselves
    (64, 32, 32, 32, 3, 1, "fp64"),
])
def test_cluster_exchange_that_runs_out_gives_nan_and_an_error(hz, monkeypatch, nx, ny, sx, sy, P, shape, precision):
    """One slab of every subdomain withholds a row that its neighbour waits for, so that the wait runs out (after
    about a second): the sweep ends with NaN in every subdomain's solution and in all that it sends, a solve with
    HZ_ERR_INTERNAL; without that, the same problem is swept and solved as ever."""
    _force(monkeypatch, shape)
    case, pr = _pair(hz, _wl(nx, ny, sx, sy, P))
    prec = hz.HZ_FP32_REFINE if precision == "fp32" else hz.HZ_FP64
    nt, lam = hz.hz_problem_nt(case.pr), _rand_lam(pr, 9)
    opts = hz.hz_default_opts(precision=prec, tol=1e-6)
    ref_l, ref_u = _run_sweep(hz, case, pr, prec, nt, 2, lam, False)
    for wh_tol in (0.0, 1e-3):
        with monkeypatch.context() as mp:
            mp.setenv("HZ_TILE_MUTE", "1")
            got_l, got_u = _run_sweep(hz, case, pr, prec, nt, 2, lam, False, wh_tol=wh_tol)
            assert np.all(np.isnan(got_u))
            assert np.all(np.isnan(got_l[lam != 0]))  # every interface slot
            if wh_tol == 0.0:
                with pytest.raises(hz.HzError) as e:
                    hz.hz_solve(case.pr, opts, n=case.n)
                assert e.value.status == hz.HZ_ERR_INTERNAL
    got_l, got_u = _run_sweep(hz, case, pr, prec, nt, 2, lam, False)
    assert np.array_equal(got_u, ref_u) and np.array_equal(got_l, ref_l)
    st, _, rep = hz.hz_solve(case.pr, opts, n=case.n)
    assert st == hz.HZ_OK and rep["rel_residual"] <= 1e-6
    case.close()


@pytest.mark.parametrize("curved", [False, True])
@pytest.mark.parametrize("nx,ny,sx,sy,P,shape", [
    (3, 3, 1, 1, 2, 1),     # 16 subdomains per warp (curved: 32)
    (12, 4, 4, 4, 3, 1),    # 2 per warp, all lanes in use
    (12, 4, 4, 4, 3, 2),    # 4 per warp
    (9, 9, 3, 3, 4, 1),     # idle lanes between the subdomains
    (16, 16, 8, 8, 3, 2),   # one subdomain per warp
])
def test_non_finite_subdomain_leaves_the_others_alone(hz, monkeypatch, nx, ny, sx, sy, P, shape, curved):
    """What one subdomain receives (NaN, infinity, a value beyond FP32) shows in its own solution and in what it
    sends, and nowhere else: every other subdomain's result is that of the clean sweep, bit for bit, also where the
    subdomains share a warp."""
    _force(monkeypatch, shape)
    case, pr = _pair(hz, _wl(nx, ny, sx, sy, P))
    if curved:
        xy = hz.hz_mesh_node_coords(case.mesh)
        xy[:, 0] += 0.02 * np.sin(np.pi * xy[:, 0]) * np.sin(np.pi * xy[:, 1])
        hz.hz_problem_set(case.pr, hz.HZ_NODE_COORDS, xy)
    nt, lam, L = hz.hz_problem_nt(case.pr), _rand_lam(pr, 10), pr.mesh.L
    ref_l, ref_u = _run_sweep(hz, case, pr, hz.HZ_FP32_REFINE, nt, 2, lam, False)
    for l in range(L):
        for value in (np.nan, np.inf, 1e300):
            bad = lam.copy()
            e = next(e for e in range(4) if pr.nbr[l, e] >= 0)
            bad[l, e, 1] = value
            got_l, got_u = _run_sweep(hz, case, pr, hz.HZ_FP32_REFINE, nt, 2, bad, False)
            others = [k for k in range(L) if k != l]
            assert not np.all(np.isfinite(got_u[l]))
            assert np.array_equal(got_u[others], ref_u[others]), (l, value)
            sent = np.zeros(lam.shape[:2], bool)  # slots that subdomain l writes
            sent[l] = pr.nbr[l] < 0
            for q in range(4):
                if pr.nbr[l, q] >= 0:
                    sent[pr.nbr[l, q], q ^ 1] = True
            assert np.array_equal(got_l[~sent], ref_l[~sent]), (l, value)
    case.close()


def test_element_ratio_rounding_does_not_build_up(hz, monkeypatch):
    """Non-square elements: (hx / hy)^2 times an assembled row that annihilates constants has to annihilate them too.
    A ratio rounded to FP32 in some of the row's terms leaves an error that every time step adds with the same sign
    (relative to the wave's own term it grows with N_t^2), where the rounding of the state grows with its square
    root.  So at a low frequency (N_t of several hundred) a badly rounded ratio, (56/79)^2, may not be worse than an
    exactly representable one, (3/4)^2, by more than the scatter of the state's rounding (a factor of 3)."""
    err = {}
    for name, ratio in (("exact", 3 / 4), ("rounded", 56 / 79)):  # hx / hy
        for shape, P in ((1, 3), (2, 3), (1, 4)):
            _force(monkeypatch, shape)
            case, pr = _pair(hz, _wl(32, 16, 16, 16, P, omega=4.0, kind="const", box=(0.0, 1.0, 0.0, 0.5 / ratio)))
            nt = hz.hz_problem_nt(case.pr)
            lam = _rand_lam(pr, 13)
            _, u = _run_sweep(hz, case, pr, hz.HZ_FP32_REFINE, nt, 8, lam, False)
            _, ref, _ = pr.sweep(lam, None, nt, 8, want_u=True)
            err[name, shape, P] = _rel(u, ref)
            case.close()
    for shape, P in ((1, 3), (2, 3), (1, 4)):
        assert err["rounded", shape, P] < 3 * err["exact", shape, P], (err, nt)
