"""The tuner's choice among the stream-collide forms (csrc/fsl_forms.h), compiled
for the host: in FP32 and 16-bit storage it stays in one family of forms whatever
the timings say, and handles of two families share no entry of the tuning cache."""
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
extern "C" int family(int prec, int multi, long long cells, int ifrac) { return family_of(prec, multi != 0, cells, ifrac); }
extern "C" int family_of_form(int form) { return form_family(form); }
extern "C" int choose(int prec, int multi, long long cells, int ifrac, const double* ms, const bool* usable) {
    return choose_form(TuneKey(prec, multi != 0, 152, cells, (cells * ifrac + 63) / 64), ms, usable);
}
extern "C" int same_key(int prec, int multi, long long a, long long ia, long long b, long long ib) {
    const TuneKey p(prec, multi != 0, 152, a, ia), q(prec, multi != 0, 152, b, ib);
    return !(p < q) && !(q < p);
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
    lib = ctypes.CDLL(so)
    i, n = ctypes.c_int, ctypes.c_longlong
    lib.family.argtypes = [i, i, n, i]
    lib.choose.argtypes = [i, i, n, i, ctypes.POINTER(ctypes.c_double), ctypes.POINTER(ctypes.c_bool)]
    lib.same_key.argtypes = [i, i, n, n, n, n]
    return lib


def choose(lib, key, ms, usable):
    return lib.choose(*key, (ctypes.c_double * FORMS)(*ms), (ctypes.c_bool * FORMS)(*usable))


def test_the_choice_stays_in_the_family_of_the_key(lib):
    rng = random.Random(3)
    for _ in range(20000):
        prec = rng.randrange(4)
        key = (prec, rng.randrange(2), int(2 ** rng.uniform(8, 27.5)), rng.randrange(0, 12))
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


# workloads on either side of the lines, as (precision, one or many domains, cells,
# interface cells in 1/64) -> first form of the family
@pytest.mark.parametrize("key, first", [
    ((F16S, 0, 199999, 8), 0), ((BF16S, 0, 200000, 8), 6), ((F16S, 0, 1 << 27, 5), 6), ((F16S, 0, 1 << 20, 1), 0),
    ((BF16S, 0, (1 << 24) - 1, 2), 0), ((F16S, 0, 1 << 24, 2), 6), ((F16S, 0, (1 << 21) - 1, 4), 0),
    ((F16S, 0, 1 << 21, 3), 6), ((F16S, 1, 199999, 8), 0), ((F16S, 1, 200000, 8), 6), ((BF16S, 1, (1 << 23) - 1, 8), 6),
    ((F16S, 1, 1 << 23, 8), 5), ((FP32, 0, (1 << 18) - 1, 8), 0), ((FP32, 0, 1 << 18, 8), 6),
    ((FP32, 0, (1 << 20) - 1, 5), 6), ((FP32, 0, 1 << 20, 5), 5), ((FP32, 0, 1 << 20, 6), 6), ((FP32, 0, 1 << 24, 5), 5),
    ((FP32, 0, (1 << 23) - 1, 3), 0), ((FP32, 0, 1 << 23, 3), 5), ((FP32, 0, 1 << 24, 1), 0),
    ((FP32, 1, (1 << 18) - 1, 8), 0), ((FP32, 1, 1 << 18, 8), 6), ((FP32, 1, 1 << 23, 8), 6)])
def test_the_families_on_either_side_of_each_line(lib, key, first):
    assert lib.family(*key) == lib.family_of_form(first)


def test_workloads_of_two_families_do_not_share_a_cached_form(lib):
    rng = random.Random(5)
    shared = 0
    for _ in range(20000):
        prec, multi, cells = rng.randrange(1, 4), rng.randrange(2), int(2 ** rng.uniform(8, 27.5))
        other, ifc = int(cells * rng.uniform(0.5, 2.0)) + 1, rng.uniform(0.0, 0.2)
        a, b = (cells, int(cells * ifc)), (other, int(other * ifc))
        if lib.same_key(prec, multi, *a, *b):
            shared += 1
            assert lib.family(prec, multi, a[0], 64 * a[1] // a[0]) == lib.family(prec, multi, b[0], 64 * b[1] // b[0])
    assert shared > 1000


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
