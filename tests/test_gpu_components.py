"""Component numbering under contention: repeated builds of one body of many
islands give the same unknowns, components and solution."""

import numpy as np
import pytest


@pytest.mark.gpu
def test_repeated_builds_of_many_islands_agree():
    torch = pytest.importorskip("torch")
    import paper_2010_12879_gb300 as spfd
    from spfd_inputs import random_phantom
    rng = np.random.default_rng(7)
    ph = random_phantom(45, 37, 29, rng, air_fraction=0.9)
    sig = torch.from_numpy(ph.sigma).cuda()
    a = torch.from_numpy(rng.normal(size=(3, 30, 38, 46))).cuda()
    first = None
    for _ in range(60):
        with spfd.Solver(sig, ph.h) as S:
            psi, info, _ = S.solve(a, 1e-6)
        got = (info["n_dof"], info["n_comp"], info["iters"])
        if first is None:
            first = (got, psi)
        assert got == first[0]
        assert torch.equal(psi, first[1])
