"""The device arrays of the step calls need the alignment of a double and no
more: views that start 8 bytes off a 16-byte boundary give, bit for bit, what
aligned arrays give (the same kernel, the same arithmetic)."""

import numpy as np
import pytest

from test_gpu_parity import _dev, _pair, _rand_lam, _wl

pytestmark = pytest.mark.gpu


def _off(t):
    """A copy of t that starts 8 bytes off a 16-byte boundary."""
    import torch

    v = torch.empty(t.numel() + 1, dtype=torch.float64, device="cuda")[1:]
    v.copy_(t)
    assert v.data_ptr() % 16 == 8
    return v


def _zeros(n, off):
    import torch

    t = torch.zeros(n, dtype=torch.float64, device="cuda")
    return _off(t) if off else t


@pytest.mark.parametrize("variant", ["tile", "warp", "block", "cluster", "cband", "curved_tile", "curved_block"])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_sweep_takes_arrays_at_any_double(hz, monkeypatch, variant, precision):
    import torch

    if precision == "fp64" and variant in ("warp", "cband", "curved_tile"):
        pytest.skip("FP32 kernels")
    monkeypatch.setenv("HZ_SWEEP_VARIANT", variant.replace("curved_", ""))
    sizes = {"tile": [(16, 16, 8, 8, 3), (32, 16, 16, 16, 4), (64, 32, 32, 32, 4)],
             "cband": [(32, 16, 16, 16, 4)]}.get(variant, [(16, 16, 8, 8, 3)])
    for size in sizes:
        wl = _wl(*size)
        case, pr = _pair(hz, wl, g_seed=3)
        if variant.startswith("curved"):
            xy = hz.hz_mesh_node_coords(case.mesh)
            x, y = xy[:, 0].copy(), xy[:, 1].copy()
            xy[:, 0] = x + 0.02 * np.sin(2 * np.pi * x) * np.sin(np.pi * y)
            xy[:, 1] = y + 0.02 * np.sin(np.pi * x) * np.sin(2 * np.pi * y)
            hz.hz_problem_set(case.pr, hz.HZ_NODE_COORDS, xy)
        nt = hz.hz_problem_nt(case.pr)
        m = pr.mesh
        prec = hz.HZ_FP32_REFINE if precision == "fp32" else hz.HZ_FP64
        rhs = _zeros(2 * case.n, False)
        hz.hz_rhs(case.pr, rhs)
        out = []
        for off in (False, True):
            lin, r = _dev(_rand_lam(pr, 4)), rhs
            if off:
                lin, r = _off(lin), _off(r)
            lout, u = _zeros(2 * m.L * 4 * m.NE, off), _zeros(2 * m.L * m.nly * m.nlx, off)
            hz.hz_sweep(case.pr, prec, nt, 2, 0.0, lin, lout, r, u)
            plain = _zeros(2 * m.L * 4 * m.NE, off)
            hz.hz_sweep(case.pr, prec, nt, 2, 0.0, lin, plain, None, None)
            total = _zeros(2 * case.n, off)
            hz.hz_assemble_add(case.pr, u, total)
            torch.cuda.synchronize()
            out.append([t.cpu().numpy() for t in (lout, u, plain, total)])
        for a, b in zip(*out):
            assert np.any(a != 0.0) and np.array_equal(a, b)
        case.close()


@pytest.mark.parametrize("nx,ny,P", [(33, 9, 3), (5, 40, 1), (20, 11, 7)])
@pytest.mark.parametrize("which", ["b", "u", "r", "all"])
def test_residual_takes_arrays_at_any_double(hz, nx, ny, P, which):
    import torch

    case, _ = _pair(hz, _wl(nx, ny, nx, ny, P))
    rng = np.random.default_rng(P)
    b, u = (_dev(rng.standard_normal(2 * case.n)) for _ in range(2))
    out = []
    for off in (False, True):
        bb, uu, r = (_off(t) if off and which in (k, "all") else t
                     for k, t in (("b", b), ("u", u), ("r", _zeros(2 * case.n, False))))
        nrm = torch.zeros(3, dtype=torch.float64, device="cuda")[1:]
        hz.hz_residual(case.pr, bb, uu, r, nrm)
        torch.cuda.synchronize()
        out.append([r.cpu().numpy(), nrm.cpu().numpy()])
    for a, c in zip(*out):
        assert np.any(a != 0.0) and np.array_equal(a, c)
    case.close()


def test_older_step_calls_take_arrays_at_any_double(hz):
    """The curved residual's u, the no-allocation residual and the lambda slot copies."""
    import torch

    wl = _wl(12, 8, 4, 4, 3)
    case, pr = _pair(hz, wl)
    m = pr.mesh
    rng = np.random.default_rng(1)
    b, u = (_dev(rng.standard_normal(2 * case.n)) for _ in range(2))
    c = torch.from_numpy(np.ascontiguousarray(case.c.ravel())).cuda()
    lam = _dev(_rand_lam(pr, 2))
    slots = torch.tensor([[0, 1], [4, 2], [m.L, 0], [2, 3]], dtype=torch.int32, device="cuda")
    out = []
    for off in (False, True):
        move = _off if off else (lambda t: t)
        r, nrm = _zeros(2 * case.n, off), _zeros(2, False)
        hz.hz_residual_noalloc(case.mesh, wl.omega, c, move(b), move(u), r, nrm)
        buf, back = _zeros(2 * 4 * m.NE, off), _zeros(lam.numel(), off)
        hz.hz_lambda_gather(case.pr, slots, 4, move(lam), buf)
        hz.hz_lambda_scatter(case.pr, slots, 4, buf, back)
        torch.cuda.synchronize()
        out.append([t.cpu().numpy() for t in (r, nrm, buf, back)])
    xy = hz.hz_mesh_node_coords(case.mesh)
    xy[:, 0] += 0.02 * np.sin(np.pi * xy[:, 0]) * np.sin(np.pi * xy[:, 1])
    hz.hz_problem_set(case.pr, hz.HZ_NODE_COORDS, xy)
    for k, off in enumerate((False, True)):
        move = _off if off else (lambda t: t)
        r, nrm = _zeros(2 * case.n, off), _zeros(2, False)
        hz.hz_residual(case.pr, move(b), move(u), r, nrm)
        torch.cuda.synchronize()
        out[k] += [r.cpu().numpy(), nrm.cpu().numpy()]
    for p, q in zip(*out):
        assert np.any(p != 0.0) and np.array_equal(p, q)
    case.close()
