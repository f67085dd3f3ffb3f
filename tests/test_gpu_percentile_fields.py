"""spfd_percentile on fields that are not spread out and with many labels: the
digits counted over the field again, the narrower ones of many labels, the
copies of a small table, and a context's scratch grown and used again with
fewer labels.  The answer is one of the inputs, so GPU and oracle are equal bit
for bit."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
SHAPE = (70, 80, 96)  # 537,600 voxels: more keys than are always listed


def _field(kind, rng):
    u = rng.random(SHAPE)
    if kind == "constant":
        return np.full(SHAPE, 0.3)
    if kind == "narrow":       # one bucket of the first digit, spread below it
        return 1.0 + 1e-3 * u
    if kind == "last_bits":    # neighbouring doubles: every digit is counted over the field
        return np.nextafter(1.0, 2.0, dtype=np.float64) + np.floor(u * 3) * 2.0 ** -52
    if kind == "ties":
        return np.floor(9 * u) * 0.7
    return np.exp(1.2 * rng.normal(size=SHAPE) - 4.0)


@pytest.fixture(scope="module")
def body():
    torch = pytest.importorskip("torch")
    import paper_2010_12879_gb300 as spfd
    from spfd_inputs import random_phantom
    ph = random_phantom(*SHAPE[::-1], np.random.default_rng(17), air_fraction=0.2)
    with spfd.Solver(torch.from_numpy(ph.sigma).cuda(), ph.h) as S:
        yield torch, S, ph.sigma


def _check(torch, S, oracle, sigma, E, lab, nlab, p):
    got, cnt = S.percentile(torch.from_numpy(E).cuda(), torch.from_numpy(lab).cuda(), nlab, p)
    want, wcnt = oracle.percentile(sigma, E, lab, nlab, p)
    assert list(cnt) == list(wcnt)
    assert np.array(got).tobytes() == np.array(want).tobytes() or np.array_equal(got, want, equal_nan=True)


@pytest.mark.parametrize("kind", ["constant", "narrow", "last_bits", "ties", "spread"])
@pytest.mark.parametrize("nlab", [0, 1, 40, 62, 63, 2048])
def test_fields_and_label_counts(body, oracle_mod, kind, nlab):
    torch, S, sigma = body
    rng = np.random.default_rng(nlab + 1)
    lab = rng.integers(-1, max(nlab, 1) + 1, SHAPE).astype(np.int32)
    if nlab > 2:
        lab[lab == 1] = 2      # an empty tissue
    _check(torch, S, oracle_mod, sigma, _field(kind, rng), lab, nlab, 0.99 if nlab % 2 else 0.37)


def test_few_many_few_labels_on_one_context(oracle_mod):
    torch = pytest.importorskip("torch")
    import paper_2010_12879_gb300 as spfd
    from spfd_inputs import random_phantom
    rng = np.random.default_rng(23)
    ph = random_phantom(40, 41, 42, rng, air_fraction=0.3)
    with spfd.Solver(torch.from_numpy(ph.sigma).cuda(), ph.h) as S:
        for nlab in (3, 127, 2048, 500, 1, 62, 3):
            E = rng.lognormal(0.0, 2.0, ph.sigma.shape)
            lab = rng.integers(0, nlab, E.shape).astype(np.int32)
            _check(torch, S, oracle_mod, ph.sigma, E, lab, nlab, 0.9)
