"""The quarter-brick kernels of small levels against the one-brick kernels.

A batch whose block orders are forced to 1 runs the one-brick kernels on
every level; single solves run the quarter-brick ones on levels of up to 512
(FP64 sweep and restriction) or 1000 bricks.  Both add their terms in the
same order, so the solutions are equal bit for bit: no tolerance is needed."""

import os
import re

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2010_12879_gb300", "csrc")


def test_pdl_early_kernels_trigger_first_and_wait():
    """Kernels launched by pdl_early() begin with pdl_trigger(), and none of
    their files lets one go without pdl_wait()."""
    names = set()
    for f in os.listdir(CSRC):
        text = open(os.path.join(CSRC, f)).read()
        names.update(re.findall(r"\bpdl_early\(\s*(k_\w+)", text))
    assert names
    for name in names:
        found = False
        for f in os.listdir(CSRC):
            text = open(os.path.join(CSRC, f)).read()
            for m in re.finditer(r"__global__[^;{]*?\b%s\s*\([^{]*\{" % name, text):
                found = True
                body = text[m.end():text.index("\n}\n", m.end())]
                first = [ln.strip() for ln in body.splitlines() if "__shared__" not in ln
                         and "constexpr" not in ln and ln.strip()][0]
                assert first == "pdl_trigger();", (name, first)
                assert "pdl_wait();" in body or "prolong_unit" in body, name
        assert found, name


@pytest.mark.gpu
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("dims,air", [((17, 9, 33), 0.3), ((40, 7, 5), 0.0), ((33, 34, 31), 0.5),
                                      ((64, 40, 100), 0.2)])
def test_quarter_bricks_equal_one_brick_kernels(dims, air, precision, monkeypatch):
    torch = pytest.importorskip("torch")
    import paper_2010_12879_gb300 as spfd
    from spfd_inputs import random_phantom
    rng = np.random.default_rng(sum(dims))
    ph = random_phantom(*dims, rng, air_fraction=air)
    nx, ny, nz = dims
    A = torch.from_numpy(rng.normal(size=(2, 3, nz + 1, ny + 1, nx + 1))).cuda()
    sig = torch.from_numpy(ph.sigma).cuda()
    prec = spfd.SPFD_MIXED if precision == "mixed" else spfd.SPFD_FP64
    monkeypatch.setenv("SPFD_TUNE_FORCE", "1")
    with spfd.Solver(sig, ph.h, precision=prec, coarse_max=64) as S:
        both, _, _ = S.solve_batch(A, 1e-9)
        for j in range(2):
            one, _, _ = S.solve(A[j].contiguous(), 1e-9)
            assert torch.equal(one, both[j])
