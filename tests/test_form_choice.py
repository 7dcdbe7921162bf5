"""The tuner's choice among the stream-collide forms (csrc/fsl_forms.h), compiled
for the host: in FP32 and 16-bit storage it stays in one family of forms whatever
the timings say, and the family depends on the key of the tuning cache only."""
import ctypes
import os
import random
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
FORMS = 9
FP64, FP32, F16S, BF16S = range(4)
SHIM = """
#include "fsl_forms.h"
using namespace fsl;
extern "C" int family(int prec, int multi, int lsize, int ifrac) { return family_of(TuneKey{prec, multi, 152, lsize, ifrac}); }
extern "C" int family_of_form(int form) { return form_family(form); }
extern "C" int choose(int prec, int multi, int lsize, int ifrac, const double* ms, const bool* usable) {
    return choose_form(TuneKey{prec, multi, 152, lsize, ifrac}, ms, usable);
}
extern "C" int cached(int form, const bool* usable) { return cached_form(form, usable); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("forms")
    (d / "shim.cpp").write_text(SHIM)
    so = str(d / "libshim.so")
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", os.path.join(ROOT, "paper_1604_01632_gb300", "csrc"),
                    "-o", so, str(d / "shim.cpp")], check=True)
    return ctypes.CDLL(so)


def choose(lib, key, ms, usable):
    return lib.choose(*key, (ctypes.c_double * FORMS)(*ms), (ctypes.c_bool * FORMS)(*usable))


def test_the_choice_stays_in_the_family_of_the_key(lib):
    rng = random.Random(3)
    for _ in range(20000):
        prec = rng.randrange(4)
        key = (prec, rng.randrange(2), rng.randrange(8, 28), rng.randrange(0, 12))
        usable = [True] * FORMS
        usable[4] = rng.random() < 0.5
        usable[6] = usable[7] = prec != FP64
        ms = [rng.uniform(0.01, 1.0) if u and rng.random() < 0.9 else 0.0 for u in usable]
        f = choose(lib, key, ms, usable)
        assert usable[f]
        family = [g for g in range(FORMS) if usable[g] and (prec == FP64 or lib.family_of_form(g) == lib.family(*key))]
        assert f in family
        timed = [ms[g] for g in family if ms[g] > 0.0]
        assert not timed or ms[f] == min(timed)


# lattices on either side of the lines, as (precision, one or many domains, log2 of
# the cells, interface cells in 1/64) -> first form of the family
@pytest.mark.parametrize("key, first", [
    ((F16S, 0, 17, 8), 0), ((BF16S, 0, 18, 8), 6), ((F16S, 0, 27, 5), 6), ((F16S, 0, 20, 1), 0), ((BF16S, 0, 23, 2), 0),
    ((F16S, 0, 24, 2), 6), ((F16S, 0, 20, 4), 0), ((F16S, 0, 21, 3), 6), ((F16S, 1, 16, 8), 0), ((F16S, 1, 17, 8), 6),
    ((BF16S, 1, 22, 8), 6), ((F16S, 1, 23, 8), 5), ((FP32, 0, 17, 8), 0), ((FP32, 0, 18, 8), 6), ((FP32, 0, 21, 5), 6),
    ((FP32, 0, 22, 5), 5), ((FP32, 0, 22, 3), 0), ((FP32, 0, 23, 3), 5), ((FP32, 0, 24, 1), 0), ((FP32, 1, 17, 8), 0),
    ((FP32, 1, 18, 8), 6), ((FP32, 1, 23, 8), 6)])
def test_the_families_on_either_side_of_each_line(lib, key, first):
    assert lib.family(*key) == lib.family_of_form(first)


def test_a_cached_slab_form_needs_the_ordered_list(lib):
    """A handle whose interface list is in appended order does not take the slab form
    that another handle of the same key left in the cache: it searches the list."""
    for order in (False, True):
        usable = (ctypes.c_bool * FORMS)(*[True] * FORMS)
        usable[4] = order
        for form in range(FORMS):
            got = lib.cached(form, usable)
            assert usable[got] and lib.family_of_form(got) == lib.family_of_form(form)
            assert got == form or (form == 4 and not order)
