"""The coarsest level's dense inverse at the edges of its forms: single-level
solves of fully conducting boxes, whose preconditioner is the inverse itself,
so that CG needs a few iterations only and Psi meets the parity bar (1e-9)."""

import numpy as np
import pytest


@pytest.mark.gpu
@pytest.mark.parametrize("dims", [(3, 3, 3),      # 64 unknowns: on the host
                                  (4, 3, 3),      # 80: one launch, five full sweeps
                                  (2, 2, 8),      # 81: a last sweep of one pivot
                                  (7, 7, 6),      # 448: seven rows per thread
                                  (7, 7, 7),      # 512: eight
                                  (8, 8, 6),      # 567: a second chunk of rows
                                  (9, 9, 9),      # 1000
                                  (9, 9, 10)])    # 1100: a launch per sweep
def test_single_level_solves(dims):
    torch = pytest.importorskip("torch")
    import oracle
    import paper_2010_12879_gb300 as spfd
    from spfd_inputs import random_phantom
    rng = np.random.default_rng(sum(dims))
    ph = random_phantom(*dims, rng, air_fraction=0.0)
    nx, ny, nz = dims
    a = rng.normal(size=(3, nz + 1, ny + 1, nx + 1))
    with spfd.Solver(torch.from_numpy(ph.sigma).cuda(), ph.h, max_levels=1) as S:
        psi, info, st = S.solve(torch.from_numpy(a).cuda(), 1e-12)
    assert st == spfd.SPFD_OK and info["n_levels"] == 1 and info["iters"] <= 6
    ref, _, sys_ = oracle.solve(ph.sigma, ph.h, a, tol=1e-13)
    g, r = oracle.project(sys_, sys_.gather(psi.cpu().numpy())), sys_.gather(ref)
    assert np.linalg.norm(g - r) <= 1e-9 * np.linalg.norm(r)
