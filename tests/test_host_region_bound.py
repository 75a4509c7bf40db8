"""The metrics' bound on a region's members, which sizes the member list.

The list's room comes from most_members (csrc/pa_regions.h), so a region may
never have more members than it says.  The header is plain C++: it is compiled
here by itself and compared with the members that the oracle's membership test
counts, over discs and annuli of sub-pixel to image size, pixels of up to 20 : 1,
centres on and off the pixel lattice.  The kernel clips its list to that room and
reports no more members than it wrote, which the source must keep doing."""

import ctypes
import os
import subprocess

import numpy as np
import pytest

from oracle import metrics as om

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2203_14906_gb300", "csrc")
SHAPES = {"rect": 0, "disc": 1, "annulus": 2}


@pytest.fixture(scope="module")
def most_members(tmp_path_factory):
    d = tmp_path_factory.mktemp("regions")
    src, lib = d / "bound.cpp", d / "bound.so"
    src.write_text('#include "pa_regions.h"\nextern "C" long long most(int s, double a, double b, int w,'
                   " int r, int inside, double dx, double dz) {"
                   " return pa::most_members(s, a, b, w, r, inside != 0, dx, dz); }\n")
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-I",
                    os.path.join(ROOT, "include"), str(src), "-o", str(lib)], check=True)
    f = ctypes.CDLL(str(lib)).most
    f.restype = ctypes.c_longlong
    f.argtypes = [ctypes.c_int, ctypes.c_double, ctypes.c_double, ctypes.c_int, ctypes.c_int,
                  ctypes.c_int, ctypes.c_double, ctypes.c_double]
    return f


def _box(c, h, o, d, n):
    """Index range of a region's box, as pa_image_metrics takes it."""
    lo = np.clip(np.floor((c - h - o) / d - 0.5) - 1, 0, n)
    hi = np.clip(np.ceil((c + h - o) / d - 0.5) + 2, 0, n)
    return int(lo), max(int(lo), int(hi))


@pytest.mark.parametrize("seed", range(6))
def test_no_region_has_more_members_than_its_room(most_members, seed):
    rng = np.random.default_rng(seed)
    tight = 0
    for _ in range(400):
        nx, nz = int(rng.integers(8, 260)), int(rng.integers(8, 260))
        dx = 10.0 ** rng.uniform(-5, -3)
        dz = dx * 10.0 ** rng.uniform(-1.3, 1.3)
        g = dict(nx=nx, nz=nz, x0_m=-0.5 * nx * dx, x1_m=0.5 * nx * dx, z0_m=0.3 * dz, z1_m=(nz + 0.3) * dz)
        gdx, gdz = (g["x1_m"] - g["x0_m"]) / nx, (g["z1_m"] - g["z0_m"]) / nz
        big = 0.5 * min(nx * dx, nz * dz)
        a = min(dx, dz) * 10.0 ** rng.uniform(-1, np.log10(max(big / min(dx, dz), 1.0)) + 0.05)
        b = a * rng.choice([0.7, 1.0, 1.02, 1.5, 3.0])
        xc = g["x0_m"] + rng.uniform(0, nx) * dx
        zc = g["z0_m"] + rng.uniform(0, nz) * dz
        if rng.random() < 0.3:  # on a pixel's centre
            xc = g["x0_m"] + (int(rng.integers(nx)) + 0.5) * gdx
            zc = g["z0_m"] + (int(rng.integers(nz)) + 0.5) * gdz
        shape = rng.choice(["disc", "annulus", "annulus"])
        r = b if shape == "annulus" else a
        j0, j1 = _box(xc, r, g["x0_m"], gdx, nx)
        l0, l1 = _box(zc, r, g["z0_m"], gdz, nz)
        inside = j0 > 0 and l0 > 0 and j1 < nx and l1 < nz
        room = most_members(SHAPES[shape], a, b, j1 - j0, l1 - l0, inside, gdx, gdz)
        have = int(om.region_mask(g, dict(shape=shape, xc_m=xc, zc_m=zc, a_m=a, b_m=b)).sum())
        assert have <= room, (shape, a / gdx, b / gdz, gdz / gdx, have, room)
        tight += inside and room < (j1 - j0) * (l1 - l0)
    assert tight > 50  # the analytic bound was the one in force


def test_the_kernel_reports_no_more_members_than_it_listed():
    src = open(os.path.join(CSRC, "pa_metrics.cu")).read()
    kernel = src[src.index("k_m_members("):src.index("struct SlotRef")]
    assert "counts[blockIdx.x] = min(run, room)" in kernel
    assert "room - off[c]" in kernel
