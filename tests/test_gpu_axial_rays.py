"""FP32 rays almost parallel to a tube's axis: transverse direction components from
1e-3 down to where their squares leave the FP32 range."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


def axial(div, rmin, x, z, n):
    """A pencil beam along z with divergence `div` from (x, 0, z), and a vacuum tube of
    radius 0.5 and half height 1 about the origin's z axis with a collar behind it."""
    return {"name": "axial", "world": {"shape": W.BOX, "centre": (0.0, 0.0, 0.0), "params": (20.0, 20.0, 20.0)},
            "prims": [W.prim(W.TUBE, (0, 0, 0), (rmin, 0.5, 1.0), axis=2)],
            "materials": [], "bias": np.zeros((0, 3)),
            "source": {"kind": "pencil", "centre": (x, 0.0, z), "half": (0.0, 0.0), "lambda": (1.8, 1.8),
                       "div": (div, div), "aperture": None},
            "tallies": [W.tally("count", "entry", 0, face=2), W.tally("count", "exit", 0, face=3),
                        W.tally("count", "exit", 0)],
            "precision": "f32", "instances": {"params": np.zeros((1, 0)), "counts": np.array([n])}, "params": [],
            "seed": 4096, "event_cap": 4096}


@pytest.mark.parametrize("kernel", [1, 2, 3])
@pytest.mark.parametrize("rmin,x", [(0.0, 0.0), (0.0, 0.3), (0.0, 1e-4), (0.2, 0.3), (1e-3, 0.4)])
@pytest.mark.parametrize("div", [0.0, 1e-38, 1e-30, 1e-24, 1e-21, 1e-20, 1e-19, 1e-18, 1e-16, 1e-15, 1e-12, 1e-3])
def test_beam_through_a_tube(div, rmin, x, kernel):
    """Every neutron enters by the front cap and leaves by the rear one: it drifts
    9e-3 * sqrt(2) cm at most, less than any margin here (0.1 cm; 0.099 of x = 0.4)."""
    from paper_2304_06226_gb300.engine import Scene
    n = 2000
    sc = Scene(axial(div, rmin, x, -8.0, n))
    sc.run(n, kernel=kernel)
    torch.cuda.synchronize()
    entered, rear, left = sc.raw()["sum"]
    cnt = sc.counters()
    sc.close()
    assert (entered, rear, left) == (n, n, n)
    assert cnt["lost"] == 0 and cnt["truncated"] == 0


@pytest.mark.parametrize("div", [1e-38, 1e-24, 1e-20, 1e-19, 1e-18, 1e-15, 1e-12, 1e-3])
@pytest.mark.parametrize("x", [0.0, 0.3])
def test_beam_from_inside_a_tube_leaves_by_its_cap(div, x):
    from paper_2304_06226_gb300.engine import Scene
    n = 2000
    sc = Scene(axial(div, 0.0, x, 0.0, n))
    sc.run(n, kernel=1)
    torch.cuda.synchronize()
    _, rear, left = sc.raw()["sum"]
    sc.close()
    assert (rear, left) == (n, n)


def test_beam_down_a_hollow_tube_misses_its_wall():
    """Along the axis inside the inner radius there is nothing to enter."""
    from paper_2304_06226_gb300.engine import Scene
    for div in (0.0, 1e-30, 1e-20, 1e-19, 1e-15):
        sc = Scene(axial(div, 0.2, 0.1, -8.0, 500))
        sc.run(500, kernel=1)
        torch.cuda.synchronize()
        assert not sc.raw()["sum"].any(), div
        sc.close()
