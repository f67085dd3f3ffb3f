"""A batch whose buffers cannot be allocated is refused with SPFD_ENOMEM and
leaves the context fit for use: the next solve, gradient, batch or group solve
allocates what is missing and gives the bits it gave before.  Device
allocations are made to fail one by one (SPFD_FAIL_ALLOC_AT)."""

import numpy as np
import pytest


@pytest.mark.gpu
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_context_survives_a_failed_batch(precision, monkeypatch):
    torch = pytest.importorskip("torch")
    import paper_2010_12879_gb300 as spfd
    from spfd_inputs import random_phantom
    rng = np.random.default_rng(41)
    ph = random_phantom(20, 17, 18, rng, air_fraction=0.4)
    sig = torch.from_numpy(ph.sigma).cuda()
    A = torch.from_numpy(rng.normal(size=(3, 3, 19, 18, 21))).cuda()
    a = A[1].contiguous()
    prec = spfd.SPFD_MIXED if precision == "mixed" else spfd.SPFD_FP64

    def build():
        return spfd.Solver(sig, ph.h, precision=prec, coarse_max=100, autotune=0)

    n0 = 1  # allocations of the build: the first one that can fail without failing it
    while True:
        monkeypatch.setenv("SPFD_FAIL_ALLOC_AT", str(n0))
        try:
            build().close()
            break
        except spfd.SpfdError as e:
            assert e.status == spfd.SPFD_ENOMEM
        n0 += 1
    monkeypatch.delenv("SPFD_FAIL_ALLOC_AT")
    refused = 0
    for n in range(n0, n0 + 80):
        with build() as S, spfd.Group([S]) as G:
            one = S.solve(a, 1e-9)[0].clone()
            (grp,), _, _ = G.solve([a], 1e-9)
            monkeypatch.setenv("SPFD_FAIL_ALLOC_AT", str(n))
            try:
                S.solve_batch(A, 1e-9)
                failed = False
            except spfd.SpfdError as e:
                failed = True
                assert e.status == spfd.SPFD_ENOMEM
            monkeypatch.delenv("SPFD_FAIL_ALLOC_AT")
            if not failed:
                break
            refused += 1
            if refused % 3 == 0:
                assert torch.equal(S.solve(a, 1e-9)[0], one)
            elif refused % 3 == 1:
                assert torch.equal(G.solve([a], 1e-9)[0][0], grp)
            else:
                J, _, _, _, st = S.energy_grad(a, one, 1.0, 1e-9)
                assert st == spfd.SPFD_OK and J > 0
            assert torch.equal(S.solve_batch(A, 1e-9)[0][1], one)
            assert torch.equal(S.solve(a, 1e-9)[0], one)
            assert torch.equal(G.solve([a], 1e-9)[0][0], grp)
    assert not failed and refused >= 10
