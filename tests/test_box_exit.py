"""The way out of a box (csrc/tp_box_exit.h), compiled for the host, against the
plain form: per axis (+-p - q) / v, the smallest, axes with v = 0 left out."""
import ctypes as C
import subprocess
from pathlib import Path

import numpy as np
import pytest

ROOT = Path(__file__).resolve().parent.parent


@pytest.fixture(scope="module")
def box_exit(tmp_path_factory):
    d = tmp_path_factory.mktemp("box_exit")
    (d / "b.cpp").write_text('#include "tp_box_exit.h"\nextern "C" double box_exit(const double* p, const double* q, '
                             'const double* v, int* f) { return tp::box_exit(p, q, v, INFINITY, f); }\n')
    subprocess.run(["g++", "-O2", "-shared", "-fPIC", f"-I{ROOT / 'paper_2304_06226_gb300' / 'csrc'}",
                    str(d / "b.cpp"), "-o", str(d / "b.so")], check=True)
    lib = C.CDLL(str(d / "b.so"))
    lib.box_exit.restype = C.c_double

    def call(p, q, v):
        f = C.c_int(-9)
        return lib.box_exit((C.c_double * 3)(*p), (C.c_double * 3)(*q), (C.c_double * 3)(*v), C.byref(f)), f.value
    return call


def plain(p, q, v):
    best, face = np.inf, -1
    for a in range(3):
        if v[a] != 0:
            t = ((p[a] if v[a] > 0 else -p[a]) - q[a]) / v[a]
            if t < best:
                best, face = t, 2 * a + (v[a] > 0)
    return best, face


@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("side", [-1.0, 1.0])
@pytest.mark.parametrize("zero", [0.0, -0.0])
def test_a_face_the_ray_is_parallel_to_is_no_exit(box_exit, axis, side, zero):
    """Also where the point lies a rounding beyond that face."""
    p = [1.0, 2.0, 3.0]
    for beyond in (0.5, 1.0, 1.0 + 2.0 ** -52, 1.0 + 1e-9):
        q, v = [0.1, -0.2, 0.3], [0.6, 0.5, -0.4]
        q[axis], v[axis] = side * beyond * p[axis], zero
        assert box_exit(p, q, v) == plain(p, q, v)
        only = [0.0] * 3
        only[(axis + 1) % 3] = 1.0
        assert box_exit(p, q, only) == plain(p, q, only)


def test_no_direction_has_no_exit(box_exit):
    assert box_exit([1, 1, 1], [0, 0, 2], [0.0, -0.0, 0.0]) == (np.inf, -1)


def test_random_rays_leave_where_the_plain_form_says(box_exit):
    """The chosen quotient is the plain form's own, bit for bit; at an edge, where
    two faces are within a rounding of one another, it may be the other one."""
    rng = np.random.Generator(np.random.PCG64(5))
    other = 0
    for i in range(20_000):
        scale = 10.0 ** rng.uniform(-3, 6)
        p = scale * rng.uniform(0.01, 1.0, 3)
        q = rng.uniform(-1, 1, 3) * p
        v = rng.normal(size=3) * 10.0 ** rng.uniform(-12, 0, 3) ** (i % 2)
        v /= np.linalg.norm(v)
        v[rng.integers(0, 3)] *= (i % 5 != 0)
        t, f = box_exit(p, q, v)
        t0, f0 = plain(p, q, v)
        if f != f0:
            other += 1
            assert abs(t - t0) <= 4 * np.spacing(t0)
        else:
            assert t == t0
    assert other == 0   # none of these seeded rays meets an edge
