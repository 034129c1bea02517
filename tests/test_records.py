"""The packed records of the batched factorisation (csrc/records.cpp), executed on
the CPU with the marks of finished pivots that the kernels read."""
import ctypes as C
import os
import subprocess
import tempfile

import numpy as np
import pytest

from paper_1711_10579_gb300 import build, cases

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1711_10579_gb300", "csrc")


@pytest.fixture(scope="module")
def host():
    so = os.path.join(tempfile.mkdtemp(prefix="records"), "records_host.so")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-shared", "-fPIC",
                           "-I", os.path.join(build._cuda_home(), "include"), "-o", so,
                           os.path.join(HERE, "records_host.cpp"),
                           *[os.path.join(CSRC, f) for f in ("records.cpp", "symbolic.cpp")]])
    return C.CDLL(so)


@pytest.mark.parametrize("by_work", [0, 1])
@pytest.mark.parametrize("ilu", [0, 1])
@pytest.mark.parametrize("n", [1, 2, 14, 33, 300, 2000])
def test_records_with_early_inverses_factor_the_matrix(host, n, ilu, by_work):
    """L U = A on the pattern of a diagonally dominant random matrix to a few ulps
    of a row's sum; unsorted, a level's items are in the order of the entries
    (neighbours in memory), which the kernels without sorted records rely on for
    their speed."""
    if n > 2:
        g = cases.transmission_case(n, int(1.35 * n), max(1, n // 5), 3, max_angle=0.06)
        f, t = (np.ascontiguousarray(a, np.int32) for a in (g.br_from, g.br_to))
    else:
        f, t = np.arange(n - 1, dtype=np.int32), np.arange(1, n, dtype=np.int32)
    err, descents = C.c_double(-1.0), C.c_int(-1)
    rc = host.records_check(n, len(f), f.ctypes.data_as(C.c_void_p), t.ctypes.data_as(C.c_void_p),
                            ilu, by_work, C.byref(err), C.byref(descents))
    assert rc == 0
    assert 0.0 <= err.value <= 1e-12
    if not by_work:
        assert descents.value == 0


def test_served_records_are_in_the_order_of_the_entries():
    """The records the library uploads for every other kernel (pf_schedule)."""
    from paper_1711_10579_gb300 import pf

    case = cases.transmission_case(300, 405, 60, 2)
    sch = pf.pf_schedule(case)
    for a, b in zip(sch["fac_ptr"][:-1], sch["fac_ptr"][1:]):  # by pivot, then by row
        e, k = sch["fac_rec"][a:b, 0], sch["fac_rec"][a:b, 1]
        assert np.array_equal(np.lexsort((e, k)), np.arange(b - a))
    for a, b in zip(sch["tgt_ptr"][:-1], sch["tgt_ptr"][1:]):
        assert np.all(np.diff(sch["tgt_rec"][a:b, 0] & ~(1 << 30)) > 0)
