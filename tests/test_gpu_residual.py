"""The residual at the edges of its blocks (32 element columns by 4 node rows, 128 rows of the last
node column) against the oracle's matrix-free K; 1e-12, the bound of
test_rhs_residual_assembly_match_oracle (the same sums in another order)."""

import numpy as np
import pytest

from test_gpu_parity import _dev, _host_c, _pair, _rel, _wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,P", [(1, 1, 3), (31, 5, 2), (32, 4, 3), (33, 9, 4), (64, 33, 1), (5, 40, 7)])
def test_residual_at_block_edges_matches_oracle(hz, nx, ny, P):
    import torch

    case, pr = _pair(hz, _wl(nx, ny, nx, ny, P, box=(-0.5, 1.5, 0.25, 1.0)), g_seed=P)
    rng = np.random.default_rng(P)
    u, b = (rng.standard_normal(case.n) + 1j * rng.standard_normal(case.n) for _ in range(2))
    r = torch.empty(2 * case.n, dtype=torch.float64, device="cuda")
    nrm = torch.empty(2, dtype=torch.float64, device="cuda")
    for bb in (b, None):
        hz.hz_residual(case.pr, None if bb is None else _dev(bb), _dev(u), r, nrm)
        ref = (0 if bb is None else bb) - pr.apply_K(u.reshape(pr.c.shape)).ravel()
        assert _rel(_host_c(r), ref) < 1e-12
        n2 = nrm.cpu().numpy()
        assert abs(n2[0] - np.sum(np.abs(ref) ** 2)) < 1e-10 * n2[0]
        assert n2[1] == 0.0 if bb is None else abs(n2[1] - np.sum(np.abs(b) ** 2)) < 1e-12 * n2[1]
    case.close()
