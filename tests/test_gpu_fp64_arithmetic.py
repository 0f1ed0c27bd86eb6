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
