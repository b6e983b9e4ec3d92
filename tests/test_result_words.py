"""Results of the kernels that count a plan on their own, as the host reads
them back: totals and busy cycles, and an error word that fails the call (no
input reaches it: a set never holds more than the largest degree)."""

import ctypes
import os
import subprocess

import pytest

from paper_2009_10955_gb300 import _native, build

SOURCE = """
#include <cstdarg>
#include <cstring>
#include "bits.cuh"
void gp::set_error(const char*, ...) {}
extern "C" int status(int n, const unsigned long long* totals, const int* errs, unsigned long long* out,
                      unsigned long long* busy) {
    gp::ResultWords words[8];
    uint64_t* res[8];
    std::memset(words, 0, sizeof(words));
    for (int j = 0; j < n; ++j) {
        words[j].total[0] = totals[2 * j];
        words[j].total[1] = totals[2 * j + 1];
        words[j].busy = 10 + j;
        words[j].err = errs[j];
        res[j] = (uint64_t*)out + 2 * j;
    }
    uint64_t b = 0;
    const int rc = gp::read_results(words, n, res, &b);
    *busy = b;
    return rc;
}
"""


@pytest.fixture(scope="module")
def status(tmp_path_factory):
    d = tmp_path_factory.mktemp("words")
    (d / "words.cu").write_text(SOURCE)
    so = str(d / "words.so")
    subprocess.run([build._nvcc(), build.ARCH, "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I" + build.CSRC,
                    "-I" + os.path.join(build.ROOT, "include"), "-o", so, str(d / "words.cu")], check=True)
    return ctypes.CDLL(so).status


@pytest.mark.parametrize("errs", [[0], [0, 0, 0], [1], [0, 0, 3], [2, 0, 0]])
def test_error_word_fails_the_call(status, errs):
    n = len(errs)
    totals = (ctypes.c_ulonglong * (2 * n))(*range(1, 2 * n + 1))
    out, busy = (ctypes.c_ulonglong * (2 * n))(), ctypes.c_ulonglong()
    rc = status(n, totals, (ctypes.c_int * n)(*errs), out, ctypes.byref(busy))
    if any(errs):
        assert rc == _native.GP_ERR_INTERNAL
    else:
        assert (rc, list(out), busy.value) == (0, list(totals), sum(range(10, 10 + n)))
