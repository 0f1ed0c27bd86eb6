"""FP64 arithmetic of the transport kernels against 64-bit values worked out here."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu

KERNELS = [1, 2, 3]


def inside_a_box(sigma):
    """A pencil beam along z from the origin, inside a large box of one scatterer."""
    return {"name": "inside", "world": {"shape": W.BOX, "centre": (0.0, 0.0, 0.0), "params": (600.0,) * 3},
            "prims": [W.prim(W.BOX, (0, 0, 0), (500.0,) * 3, material=0)],
            "materials": [W.material(sigma_inc=sigma)], "bias": np.ones((1, 3)),
            "source": {"kind": "pencil", "centre": (0.0, 0.0, 0.0), "half": (0.0, 0.0), "lambda": (1.8, 1.8),
                       "div": (0.0, 0.0), "aperture": None},
            "tallies": [W.tally("count", "exit", 0)], "precision": "f64",
            "instances": {"params": np.zeros((1, 0)), "counts": np.array([1])}, "params": [], "seed": 4096,
            "event_cap": 4096}


def first_flights(sigma, kernel, n=50_000):
    from paper_2304_06226_gb300.engine import Scene, new_records, records_to_numpy
    sc, rec = Scene(inside_a_box(sigma)), new_records(n)
    sc.run(n, kernel=kernel, records=rec)
    torch.cuda.synchronize()
    sc.close()
    return records_to_numpy(rec)["first_collision"][:, 2]


@pytest.mark.parametrize("sigma", [0.3, 0.7, 1.1, 3.0])
@pytest.mark.parametrize("kernel", KERNELS)
def test_flight_length_is_a_correctly_rounded_quotient(kernel, sigma):
    """The first collision lies at -log(xi) / Sigma beyond the origin, to the last
    bit: a cross section of 1 gives -log(xi) itself, and IEEE division the rest."""
    z1, z = first_flights(1.0, kernel), first_flights(sigma, kernel)
    assert np.isfinite(z1).all()
    assert (z == z1 / sigma).all(), (z != z1 / sigma).mean()


def escape_angles(scale, bins, lo, hi, axis, off):
    """Isotropic scatter in a sphere of radius `scale`, counted by angle on a world
    sphere a hundred times as large."""
    d = inside_a_box(1.0 / scale)
    d["world"] = {"shape": W.SPHERE, "centre": (0.0, 0.0, 0.0), "params": (0.0, 100.0 * scale, 0.0)}
    d["prims"] = [W.prim(W.SPHERE, (0, 0, 0), (0.0, scale, 0.0), material=0)]
    d["source"]["centre"] = (0.0, 0.0, -10.0 * scale)
    d["tallies"] = [W.tally("angular", "exit", -1, bins=(bins, 1), lo=(lo, 0.0), hi=(hi, 1.0),
                            origin=tuple(off * scale * k for k in (1, -2, 3)), axis=axis)]
    return d


@pytest.mark.parametrize("scale", [1e-3, 1.0, 1e6, 1e15, 1e17, 1e18, 1e19, 1e22, 1e40])
@pytest.mark.parametrize("bins,lo,hi,axis,off", [(180, 0.0, np.pi, (0, 0, 1), 0.0), (3601, 0.0, np.pi, (0, 0, 1), 0.0),
                                                 (1237, 0.3, 1.7, (1, 2, -2), 0.1), (100_003, 0.0, 3.2, (0, -3, 0), 0.7),
                                                 (1, 1.0, 1.5, (1, 0, 0), 0.0)])
def test_angular_bins_are_those_of_the_64_bit_angle(scale, bins, lo, hi, axis, off):
    """Every history's bin from the recorded end of its path: the tally holds the
    same counts (an angle within rounding of an edge, some 1e-15 of a radian, does
    not occur among 1e5)."""
    from paper_2304_06226_gb300.engine import Scene, new_records, records_to_numpy
    n = 100_000
    d = escape_angles(scale, bins, lo, hi, axis, off)
    sc, rec = Scene(d), new_records(n)
    sc.run(n, kernel=3, records=rec)
    torch.cuda.synchronize()
    got, x = sc.raw()["sum"], records_to_numpy(rec)["final_pos"]
    sc.close()
    assert (np.abs(x).max(axis=1) > scale).all()
    v = (x - d["tallies"][0]["origin"]) / scale
    a = np.asarray(axis) / np.linalg.norm(axis)
    th = np.arctan2(np.linalg.norm(np.cross(v, a), axis=1), v @ a)
    b = np.floor((th - lo) * (bins / (hi - lo))).astype(np.int64)
    want = np.bincount(b[(th >= lo) & (th < hi)], minlength=bins)
    assert want.sum() > n // 20
    assert (got == want[:bins]).all(), np.abs(got - want[:bins]).sum()
