"""The autotuner keeps, beside the fastest sweep kernel of a shape, the fastest one that reads a start (register-resident
bands or the block kernel), and warm-started sweeps run that one; what it keeps for one kind of problem (square elements
or not, interface boundary mass or not) is not taken for another."""

import re

import numpy as np
import pytest

from test_gpu_parity import _pair, _wl

pytestmark = pytest.mark.gpu


def _tuned(log):
    """{key: [(variant, configuration, ms)]} of HZ_TUNE_LOG."""
    out = {}
    for key, v, t, ms in re.findall(r"hz autotune (\S+): candidate (\d+)/(\d+) ([0-9.]+) ms", log):
        out.setdefault(key, []).append((int(v), int(t), float(ms)))
    return out


@pytest.mark.parametrize("precision,layout", [("fp32", (24, 24, 8, 8, 3)), ("fp32", (20, 20, 5, 5, 3)),
                                              ("fp64", (24, 24, 8, 8, 3))])
def test_warm_start_runs_the_fastest_kernel_that_reads_it(hz, monkeypatch, capfd, precision, layout):
    monkeypatch.setenv("HZ_TUNE_LOG", "1")
    prec = hz.HZ_FP32_REFINE if precision == "fp32" else hz.HZ_FP64
    # boxes and frequency of its own: nothing in the process has tuned this shape before
    case, pr = _pair(hz, _wl(*layout, omega=6.0, kind="const", box=(0.0, 1.3, 0.0, 0.9)))
    capfd.readouterr()
    opts = dict(precision=prec, tol=1e-2, outer=hz.HZ_OUTER_PLAIN, wh_iters=20, wh_tol=1e-3, max_sweeps=400, autotune=1)
    _, _, rep = hz.hz_solve(case.pr, hz.hz_default_opts(wh_warm=1, **opts), n=case.n)
    log = _tuned(capfd.readouterr().err)
    assert len(log) == 1
    readers = [c for c in next(iter(log.values())) if c[0] in (1, 2)]  # block, warps
    assert readers
    best = min(readers, key=lambda c: c[2])
    near = [c for c in readers if c[2] <= 1.001 * best[2]]  # the log's digits may hide which of two equals it was
    assert (rep["sweep_variant"], rep["sweep_shape"]) in [c[:2] for c in near], (rep, log)
    case.close()


def test_tuned_kernels_of_square_and_other_elements_and_of_eta_are_kept_apart(hz, monkeypatch, capfd):
    monkeypatch.setenv("HZ_TUNE_LOG", "1")
    keys = set()
    for box, eta in (((0.0, 1.0, 0.0, 1.0), 0.0), ((0.0, 1.0, 0.0, 0.7), 0.0), ((0.0, 1.0, 0.0, 1.0), 0.2)):
        case, pr = _pair(hz, _wl(12, 12, 6, 6, 2, box=box), robin=(eta, 1.0))
        capfd.readouterr()
        hz.hz_solve(case.pr, hz.hz_default_opts(precision=hz.HZ_FP32_REFINE, tol=1e-3, autotune=1), n=case.n)
        log = _tuned(capfd.readouterr().err)
        assert len(log) == 1 and not set(log) & keys, (box, eta)
        tiles = [c for c in next(iter(log.values())) if c[0] == 7]
        assert bool(tiles) == (eta == 0.0)
        keys |= set(log)
        case.close()
