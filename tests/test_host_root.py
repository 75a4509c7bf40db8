"""The envelope's square root has sqrtf's bits or is marked as undecided.

csrc/pa_root.h is plain C++ beside device code: it is compiled here with estimates
of the reciprocal root anywhere within the device instruction's documented error
(2^-22.9, relative) and compared with the correctly rounded root: dense runs of
floats, both octave parities, the ends of its range, and squares and their
neighbours, next to which no midpoint lies, as well as squares of midpoints."""

import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2203_14906_gb300", "csrc")

SRC = """
#include <cmath>
#include <cstdint>
#include <cstring>
#include "pa_root.h"
extern "C" void roots(const float* v, const double* e, long n, long* wrong, long* marked) {
  *wrong = *marked = 0;
  for (long i = 0; i < n; ++i) {
    uint32_t d = 0;
    const float s = pa::root_or_mark(v[i], (float)((1.0 + e[i]) / std::sqrt((double)v[i])), d);
    if (d) ++*marked;
    else if (s != std::sqrt(v[i])) ++*wrong;
  }
}
extern "C" void range(uint32_t* lo, uint32_t* span) { *lo = pa::kRootLo; *span = pa::kRootSpan; }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("root")
    (d / "root.cpp").write_text(SRC)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC,
                    str(d / "root.cpp"), "-o", str(d / "root.so")], check=True)
    return ctypes.CDLL(str(d / "root.so"))


def _counts(lib, v, e):
    v, e = np.ascontiguousarray(v, np.float32), np.ascontiguousarray(np.broadcast_to(e, v.shape), np.float64)
    wrong, marked = ctypes.c_long(), ctypes.c_long()
    lib.roots(v.ctypes.data_as(ctypes.c_void_p), e.ctypes.data_as(ctypes.c_void_p), ctypes.c_long(v.size),
              ctypes.byref(wrong), ctypes.byref(marked))
    return wrong.value, marked.value


def test_range(lib):
    lo, span = ctypes.c_uint32(), ctypes.c_uint32()
    lib.range(ctypes.byref(lo), ctypes.byref(span))
    ends = np.array([lo.value, lo.value + span.value], np.uint32).view(np.float32)
    assert list(ends) == [2.0 ** -101, 2.0 ** 101]


# the float rounding of the estimate itself (2^-24) is part of the error
EDGE = 2.0 ** -22.9 - 2.0 ** -24


@pytest.mark.parametrize("scale", [2.0 ** -101, 2.0 ** -100, 2.0 ** -60, 0.25, 0.5, 2.0 ** 40, 2.0 ** 99])
def test_bits_of_sqrt_or_marked(lib, scale):
    rng = np.random.default_rng(3)
    n = 1 << 20
    m = np.concatenate([np.arange(n, dtype=np.float64), rng.integers(0, 1 << 23, n),  # dense, random
                        (1 << 23) - 1 - np.arange(n)])
    v = ((1.0 + m / (1 << 23)) * scale).astype(np.float32)
    for e in (0.0, EDGE, -EDGE, rng.uniform(-EDGE, EDGE, v.size)):
        wrong, marked = _counts(lib, v, e)
        assert wrong == 0
        assert marked <= 2e-5 * v.size


def test_next_to_midpoints(lib):
    """Roots nearest to midpoints of floats: squares of midpoints, rounded to floats."""
    k = np.arange(1 << 23, (1 << 23) + (1 << 21), dtype=np.float64) + 0.5
    k = np.concatenate([k, np.arange((1 << 24) - (1 << 21), 1 << 24, dtype=np.float64) - 0.5])
    v = (k * k).astype(np.float32)
    v = np.concatenate([v, np.nextafter(v, np.float32(0)), np.nextafter(v, np.float32(np.inf))])
    rng = np.random.default_rng(4)
    for e in (0.0, EDGE, -EDGE, rng.uniform(-EDGE, EDGE, v.size)):
        assert _counts(lib, v, e)[0] == 0
