"""Source check of the kernels launched by pdl_early(): they run ahead of the
kernel before them and may read only what no kernel of a solve writes until
they wait.  Each one (with the device function it hands its work to) triggers
first, waits exactly once, has no return and no access to a vector argument
before the wait, and takes its vectors without __restrict__, which would let
the compiler move their loads in front of it."""

import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2010_12879_gb300", "csrc")
TEXT = {p: re.sub(r"//[^\n]*", "", open(p).read())
        for p in sorted(glob.glob(os.path.join(CSRC, "*.cu*")))}
# kernel -> the vectors of the solve among its arguments
VECTORS = {"k_slab27": ("x", "b", "out"), "k_slab_restrict": ("rf", "bc", "xc"),
           "k_prolong": ("ec", "ef"), "k_coarse_solve": ("b", "x")}
UNITS = {"k_prolong": "prolong_unit"}


def _function(name, kind):
    """(parameters, body) of the one definition of a function."""
    found = []
    for text in TEXT.values():
        for m in re.finditer(r"%s[^;{}]*?\b%s\s*\(([^{;]*)\)\s*\{" % (kind, name), text):
            depth, i = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(text[i], 0)
                i += 1
            found.append((m.group(1), text[m.end():i - 1]))
    assert len(found) == 1, (name, len(found))
    return found[0]


def _check(params, body, vectors):
    assert body.count("pdl_wait();") == 1
    before = body[:body.index("pdl_wait();")]
    # the wait is a statement of the function's own block
    assert before.count("{") == before.count("}")
    assert not re.search(r"(if|else|for|while)\b[^;{}]*$", before)
    assert not re.search(r"\breturn\b", re.sub(r"\[[^\]]*\]\s*\([^)]*\)\s*\{[^{}]*\}", "", before))
    for v in vectors:
        assert re.search(r"[\s*]%s\s*(,|$)" % v, params.strip()), v
        assert not re.search(r"__restrict__\s+%s\s*(,|$)" % v, params.strip()), v
        assert not re.search(r"(?<![\w.])%s\s*\[|\*\s*%s\b(?!\s*\w*\s*=)|ld\w*\([^;]*\b%s\b" % (v, v, v),
                             before), v


def test_every_early_kernel_is_listed():
    launched = set()
    for text in TEXT.values():
        launched.update(re.findall(r"\bpdl_early\(\s*(k_\w+)", text))
    assert launched == set(VECTORS)


@pytest.mark.parametrize("name", sorted(VECTORS))
def test_early_kernels_touch_vectors_after_the_wait_only(name):
    params, body = _function(name, "__global__")
    first = [ln.strip() for ln in body.splitlines()
             if ln.strip() and "__shared__" not in ln and "constexpr" not in ln][0]
    assert first == "pdl_trigger();"
    if name in UNITS:
        assert "pdl_wait" not in body and body.count(UNITS[name] + "<") == 1
        assert not re.search(r"\breturn\b", body)
        for v in VECTORS[name]:
            assert not re.search(r"\b%s\s*\[" % v, body)
            assert not re.search(r"__restrict__\s+%s\s*(,|$)" % v, params.strip())
        params, body = _function(UNITS[name], "__device__")
    _check(params, body, VECTORS[name])


def test_the_check_notices_what_it_is_for():
    params, body = _function("k_slab27", "__global__")
    good = ("x", "b", "out")
    _check(params, body, good)
    bad = [(params, body.replace("pdl_wait();", "")),
           (params, body.replace("pdl_wait();", "if (t < 64) pdl_wait();")),
           (params, body.replace("pdl_wait();", "if (bk > 9) return;\n  pdl_wait();")),
           (params, body.replace("pdl_wait();", "const T early = x[t];\n  pdl_wait();")),
           (params.replace("const T *x", "const T *__restrict__ x"), body)]
    for p, b in bad:
        with pytest.raises(AssertionError):
            _check(p, b, good)
