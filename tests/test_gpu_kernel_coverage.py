"""Sweep kernels that the size rules no longer take by themselves, and shapes of the element tiles that other tests reach
only with non-square elements or with a source, against the FP64 oracle (the bounds of tests/_tolerances.py).  Also that
a solve's report tells the kernels apart."""

import numpy as np
import pytest

import _tolerances as _tol
import test_gpu_warm as _warm
from _tolerances import FP32_REL
from test_gpu_parity import LAYOUTS, _dev, _host_c, _pair, _rand_lam, _rel, _run_sweep, _wl

pytestmark = pytest.mark.gpu

TILES = [(3, 3, 1, 1, 2), (12, 4, 4, 4, 3), (16, 16, 8, 8, 3), (10, 12, 5, 6, 2), (7, 9, 7, 3, 4), (16, 8, 8, 8, 1),
         (6, 4, 2, 2, 5), (24, 22, 12, 22, 3), (32, 24, 32, 24, 3)]


@pytest.mark.parametrize("nx,ny,sx,sy,P", LAYOUTS)
def test_column_kernel_matches_oracle(hz, monkeypatch, nx, ny, sx, sy, P):
    """One warp per subdomain by node columns (warm starts, interface boundary mass, packed launches) where compiled."""
    monkeypatch.setenv("HZ_SWEEP_WARPS", "1")
    case, pr = _pair(hz, _wl(nx, ny, sx, sy, P), g_seed=P)
    nt, lam = hz.hz_problem_nt(case.pr), _rand_lam(pr, 2)
    for with_rhs in (True, False):
        got_l, got_u = _run_sweep(hz, case, pr, hz.HZ_FP32_REFINE, nt, 5, lam, with_rhs)
        ref_l, ref_u, _ = pr.sweep(lam, pr.rhs() if with_rhs else None, nt, 5, want_u=True)
        assert _rel(got_u, ref_u) < FP32_REL and _rel(got_l, ref_l) < FP32_REL
    case.close()


@pytest.mark.parametrize("shape", [1, 2])
@pytest.mark.parametrize("nx,ny,sx,sy,P", TILES)
def test_tiles_of_square_elements_match_oracle(hz, monkeypatch, nx, ny, sx, sy, P, shape):
    """The instantiations for square elements, fixed count (odd and even N_t) and tolerance."""
    if shape == 2 and (sy % 2 or P > 3):
        pytest.skip("paired tiles need an even number of element rows and P <= 3")
    monkeypatch.setenv("HZ_SWEEP_VARIANT", "tile")
    monkeypatch.setenv("HZ_TILE_SHAPE", str(shape))
    case, pr = _pair(hz, _wl(nx, ny, sx, sy, P, box=(0.0, nx / 16, 0.0, ny / 16)), g_seed=nx + P)
    lam, bound = _rand_lam(pr, 5), _tol.fp32_bound(sx * P + 1)
    for nt in (hz.hz_problem_nt(case.pr), hz.hz_problem_nt(case.pr) + 1):
        for with_rhs in (True, False):
            got_l, got_u = _run_sweep(hz, case, pr, hz.HZ_FP32_REFINE, nt, 4, lam, with_rhs)
            ref_l, ref_u, _ = pr.sweep(lam, pr.rhs() if with_rhs else None, nt, 4, want_u=True)
            assert _rel(got_u, ref_u) < bound and _rel(got_l, ref_l) < bound, (nt, with_rhs)
    for with_rhs in (True, False):
        _, u = _run_sweep(hz, case, pr, hz.HZ_FP32_REFINE, nt, 30, lam, with_rhs, wh_tol=1e-3)
        _, ref_u, _ = pr.sweep(lam, pr.rhs() if with_rhs else None, nt, 30, wh_tol=1e-3, want_u=True)
        assert _rel(u, ref_u) < 1e-2, with_rhs
    if P <= 4 and shape == 1:
        got_l, got_u = _run_sweep(hz, case, pr, hz.HZ_FP64, nt, 2, lam, False)
        ref_l, ref_u, _ = pr.sweep(lam, None, nt, 2, want_u=True)
        assert _rel(got_u, ref_u) < 1e-12 and _rel(got_l, ref_l) < 1e-12
    case.close()


@pytest.mark.parametrize("rows", ["0", "4"])
def test_fp64_cluster_kernel_at_129_nodes(hz, monkeypatch, rows):
    monkeypatch.setenv("HZ_SWEEP_VARIANT", "cluster")
    monkeypatch.setenv("HZ_CLUSTER_TY", rows)
    case, pr = _pair(hz, _wl(64, 32, 32, 32, 4))
    nt, lam = hz.hz_problem_nt(case.pr), _rand_lam(pr, 6)
    got_l, got_u = _run_sweep(hz, case, pr, hz.HZ_FP64, nt, 1, lam, False)
    ref_l, ref_u, _ = pr.sweep(lam, None, nt, 1, want_u=True)
    assert _rel(got_u, ref_u) < 1e-12 and _rel(got_l, ref_l) < 1e-12
    case.close()


@pytest.mark.parametrize("nx,ny,sx,sy,P", [(12, 4, 4, 4, 3), (16, 16, 8, 8, 3)])
def test_warm_start_on_curved_tiles(hz, monkeypatch, nx, ny, sx, sy, P):
    import torch

    monkeypatch.setenv("HZ_SWEEP_VARIANT", "tile")
    case, pr = _warm._case(hz, nx, ny, sx, sy, P, amp=0.04)
    m, nt, lam = pr.mesh, hz.hz_problem_nt(case.pr), _warm._lam(pr, 3)
    rng = np.random.default_rng(4)
    u0 = rng.standard_normal((m.L, m.nly, m.nlx)) + 1j * rng.standard_normal((m.L, m.nly, m.nlx))
    ref_l, ref_u, _ = pr.sweep(lam, None, nt, 2, want_u=True, u0=u0)
    lout = torch.zeros(2 * hz.hz_lambda_size(case.pr), dtype=torch.float64, device="cuda")
    u = _dev(u0)
    hz.hz_sweep_from(case.pr, hz.HZ_FP32_REFINE, nt, 2, 0.0, _dev(lam), lout, None, u, u)
    torch.cuda.synchronize()
    assert _rel(_host_c(u).reshape(ref_u.shape), ref_u) < FP32_REL
    assert _rel(_host_c(lout).reshape(ref_l.shape), ref_l) < FP32_REL
    case.close()


def test_reports_tell_the_kernels_apart(hz, monkeypatch):
    seen = {}
    for env in ("tile1", "tile2", "warp", "block"):
        monkeypatch.setenv("HZ_SWEEP_VARIANT", env[:4] if env.startswith("tile") else env)
        monkeypatch.setenv("HZ_TILE_SHAPE", env[4:] or "0")
        case, _ = _pair(hz, _wl(16, 16, 8, 8, 3))
        _, _, rep = hz.hz_solve(case.pr, hz.hz_default_opts(precision=hz.HZ_FP32_REFINE, tol=1e-4), n=case.n)
        seen[env] = rep["sweep_variant"], rep["sweep_shape"]
        case.close()
    assert seen["tile1"] == (2, 32 + 3) and seen["tile2"] == (2, 64 + 1)
    assert seen["warp"] == (2, 1) and seen["block"][0] == 1
