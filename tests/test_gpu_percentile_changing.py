"""spfd_percentile reads |E| and the labels in several passes.  Inputs that
another stream changes during the call break its rules; the call then answers
or refuses with SPFD_EINTERNAL, reads nothing out of range, and leaves the
context fit for the next call."""

import os
import re
import threading

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2010_12879_gb300", "csrc")


def test_list_is_read_up_to_the_entries_written():
    """k_pct_hist takes its bound from the list's cursor on the device."""
    text = open(os.path.join(CSRC, "spfd_percentile.cu")).read()
    m = re.search(r"k_pct_hist\(([^{]*)\{(.*?)\n\}\n", text, re.S)
    args, body = m.groups()
    assert "unsigned long long *__restrict__ listed" in args
    assert "const unsigned long long n = min(*listed, want);" in body
    assert re.search(r"const bool in = i < n;", body)
    assert re.search(r"const int g = in \? kgrp\[i\] : 0;", body)


@pytest.mark.gpu
def test_labels_changed_during_the_call(oracle_mod, monkeypatch):
    torch = pytest.importorskip("torch")
    import paper_2010_12879_gb300 as spfd
    from spfd_inputs import random_phantom
    monkeypatch.setenv("SPFD_POISON_ALLOC", "1")
    rng = np.random.default_rng(31)
    ph = random_phantom(64, 48, 40, rng, air_fraction=0.2)
    E = rng.lognormal(-2.0, 1.2, ph.sigma.shape)
    lab = rng.integers(0, 12, ph.sigma.shape).astype(np.int32)
    Ed, good = torch.from_numpy(E).cuda(), torch.from_numpy(lab).cuda()
    want, wcnt = oracle_mod.percentile(ph.sigma, E, lab, 12, 0.9)
    with spfd.Solver(torch.from_numpy(ph.sigma).cuda(), ph.h) as S:
        live, side, stop = good.clone(), torch.cuda.Stream(), threading.Event()

        def flip():
            with torch.cuda.stream(side):
                while not stop.is_set():
                    live.fill_(-1)
                    side.synchronize()
                    live.copy_(good)
                    side.synchronize()

        th = threading.Thread(target=flip)
        th.start()
        try:
            for _ in range(200):
                try:
                    S.percentile(Ed, live, 12, 0.9)
                except spfd.SpfdError as e:
                    assert e.status == spfd.SPFD_EINTERNAL
        finally:
            stop.set()
            th.join()
        torch.cuda.synchronize()
        got, cnt = S.percentile(Ed, good, 12, 0.9)
    assert list(cnt) == list(wcnt) and got == list(want)
