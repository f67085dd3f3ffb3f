"""The coarsest level's dense inverse is one launch up to 1024 unknowns, in
strips of four columns where their blocks are resident at once and of eight
beyond (605 unknowns on 152 SMs), and a launch per 16 pivots above.  Single-
level boxes at the limits: the build's launches tell the form, and CG with the
inverse as its preconditioner meets the parity bar (1e-9) in a few iterations."""

import numpy as np
import pytest

# dims -> unknowns (nx + 1)(ny + 1)(nz + 1)
BOXES = [((1, 1, 150), 604), ((10, 10, 4), 605), ((10, 9, 6), 770), ((9, 7, 11), 960),
         ((1, 2, 170), 1026), ((7, 7, 15), 1024)]


@pytest.mark.gpu
@pytest.mark.parametrize("dims,m", BOXES)
def test_one_launch_up_to_1024_unknowns(dims, m):
    torch = pytest.importorskip("torch")
    import oracle
    import paper_2010_12879_gb300 as spfd
    from spfd_inputs import random_phantom
    rng = np.random.default_rng(m)
    ph = random_phantom(*dims, rng, air_fraction=0.0)
    nx, ny, nz = dims
    assert (nx + 1) * (ny + 1) * (nz + 1) == m
    a = rng.normal(size=(3, nz + 1, ny + 1, nx + 1))
    small = random_phantom(4, 3, 3, rng, air_fraction=0.0)     # 80 unknowns: one launch
    with spfd.Solver(torch.from_numpy(small.sigma).cuda(), ph.h, max_levels=1) as S:
        one = S.info()["launches"]
    with spfd.Solver(torch.from_numpy(ph.sigma).cuda(), ph.h, max_levels=1) as S:
        launches = S.info()["launches"]
        psi, info, st = S.solve(torch.from_numpy(a).cuda(), 1e-12)
    assert launches - one == (0 if m <= 1024 else (m + 15) // 16 - 1)
    assert st == spfd.SPFD_OK and info["n_levels"] == 1 and info["iters"] <= 6
    ref, _, sys_ = oracle.solve(ph.sigma, ph.h, a, tol=1e-13)
    g, r = oracle.project(sys_, sys_.gather(psi.cpu().numpy())), sys_.gather(ref)
    assert np.linalg.norm(g - r) <= 1e-9 * np.linalg.norm(r)
