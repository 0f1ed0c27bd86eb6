"""Runs of one scene before and after its materials, biases or parameters change,
against a scene that had the new values from the start.  FP64 on the history
kernel: every history has its own random numbers, so counters are equal and the
tallies agree to the rounding of their sums (up to 2e6 FP64 additions of like
sign, whose errors add like a random walk: 1e-11)."""
import copy

import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu

N = 20_000


def grid_scene_with_moving_radius():
    """60 primitives (a grid) and a sphere whose radius is the parameter."""
    d = W.imaging(n_prims=60, precision="f64", psd_bins=16)
    d["prims"].append(W.prim(W.SPHERE, (0.0, 0.0, 7.0), (0.0, 0.3, 0.0), material=2, bind_rmax=True))
    d["params"] = [{"kind": "radius", "target": -1}]
    d["instances"] = {"params": np.full((1, 1), 0.3), "counts": np.array([N]), "radius_nominal": 0.3}
    for m in d["materials"]:
        m["density_param"] = -1
    return d


def fresh(desc, seed=None, **kw):
    from paper_2304_06226_gb300.engine import Scene
    sc = Scene(desc)
    sc.run(N, kernel=1, seed=seed, **kw)
    torch.cuda.synchronize()
    out = sc.raw(), sc.counters()
    sc.close()
    return out


def same(sc, ref):
    raw, cnt = ref
    assert sc.counters() == cnt
    got = sc.raw()
    for k in ("sum", "sumsq"):
        assert raw[k].any()
        assert np.allclose(got[k], raw[k], rtol=1e-11, atol=1e-11 * np.abs(raw[k]).max()), k


@pytest.mark.parametrize("change", ["lines", "bias", "radius"])
def test_graph_run_after_the_tables_changed(change):
    from paper_2304_06226_gb300.engine import Scene
    old = W.powder(precision="f64") if change == "lines" else grid_scene_with_moving_radius()
    new = copy.deepcopy(old)
    if change == "lines":   # fewer Bragg lines: the sections behind them move
        new["materials"][0]["bragg"] = W.fcc_bragg_lines(dmin=1.0)
    elif change == "bias":
        new["bias"][:] = [[2.0, 2.0, 2.0], [1.0, 3.0, 1.0], [0.5, 1.0, 1.0]]
    else:
        new["instances"]["params"] = np.full((1, 1), 0.6)
    sc = Scene(old)
    sc.run(N, kernel=1, graph=True)
    if change == "lines":
        sc.set_materials(new["materials"])
    elif change == "bias":
        for m in range(3):
            sc.set_bias(m, new["bias"][m])
    else:
        sc.set_params(new["instances"]["params"])
    sc.reset()
    sc.run(N, kernel=1, graph=True)   # the same seed and counts as the first graph
    torch.cuda.synchronize()
    same(sc, fresh(new))
    sc.close()


@pytest.mark.parametrize("grid", [False, True])
def test_tables_change_behind_a_run_in_flight_on_a_side_stream(grid):
    """The first run is still on its way (some milliseconds) when the bias changes
    and the second is queued behind it: each must see its own tables."""
    from paper_2304_06226_gb300.engine import Scene
    old = W.imaging(n_prims=60, precision="f64", psd_bins=16) if grid else W.slab(g=1.0)
    m, n = len(old["materials"]), (400_000 if grid else 2_000_000)
    sc = Scene(old)
    seen = []
    for stream in (None, torch.cuda.Stream()):
        for k in range(m):
            sc.set_bias(k, old["bias"][k])
        sc.reset()
        torch.cuda.synchronize()
        sc.run(n, kernel=1, stream=stream)
        if stream is None:
            torch.cuda.synchronize()
        for k in range(m):
            sc.set_bias(k, (0.5, 3.0, 1.0))
        sc.run(1000, first=n, kernel=1, stream=stream)
        torch.cuda.synchronize()
        seen.append((sc.raw(), sc.counters()))
    same(sc, seen[0])
    sc.close()


def test_reset_runs_and_reads_on_several_streams_are_ordered():
    """Reset, two runs on two side streams, one on the default stream, the means and
    the backward pass, with no wait by the caller: what a single stream gives."""
    from paper_2304_06226_gb300.engine import Scene
    d = W.imaging(n_prims=30, precision="f64", psd_bins=64)
    sc, seen = Scene(d), []
    for streams in ((None,) * 3, (torch.cuda.Stream(), torch.cuda.Stream(), None)):
        sc.run(1000, kernel=1, want_grad=True)
        sc.reset()
        for k, (st, n) in enumerate(zip(streams, (300_000, 200_000, 100_000))):
            sc.run(n, first=10**6 * k, kernel=1, want_grad=True, stream=st)
        means = sc.means()
        with torch.cuda.stream(streams[0] or torch.cuda.default_stream()):
            grad = sc.backward(torch.ones_like(means))
        torch.cuda.synchronize()
        seen.append((means.cpu().numpy(), grad.cpu().numpy(), sc.counters()))
    sc.close()
    (m0, g0, c0), (m1, g1, c1) = seen
    assert c0 == c1 and c0["histories"] == 600_000
    assert m0.any() and np.allclose(m1, m0, rtol=1e-11, atol=1e-11 * m0.max())
    # a gradient's terms cancel: rounding against the sum of their magnitudes, below 100 a history
    assert np.allclose(g1, g0, rtol=0.0, atol=1e-9)


@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("prims", [10, 60])   # without and with a grid
def test_parameters_that_move_nothing_change_on_a_scene_that_has_run(prims, graph):
    """New densities (the geometry and its tables stay as they are), refused values
    between, then densities back: each run is that of a scene made with them."""
    from paper_2304_06226_gb300.engine import Scene
    desc = W.imaging(n_prims=prims, precision="f64", psd_bins=16)
    sc = Scene(desc)
    for dens in (None, (0.5, 2.0, 1.5), (1.0, 1.0, 1.0)):
        ref = copy.deepcopy(desc)
        if dens is not None:
            ref["instances"]["params"] = np.array([dens])
            sc.set_params(np.array([dens]))
            for bad in (np.nan, 0.0, -1.0):
                with pytest.raises(RuntimeError):
                    sc.set_params(np.array([[1.7, 1.7, bad]]))
        sc.reset()
        sc.run(N, kernel=1, graph=graph)
        torch.cuda.synchronize()
        same(sc, fresh(ref))
    sc.close()


def test_a_tally_read_on_a_side_stream_waits_for_the_work_its_buffers_come_from():
    """The buffers of a read may be memory that earlier work of the side stream, freed
    but not finished, still writes: it must not land in the result."""
    from paper_2304_06226_gb300.engine import Scene
    d = W.powder(precision="f64")
    sc = Scene(d)
    sc.run(N, kernel=1)
    torch.cuda.synchronize()
    want = sc.tally(0)[0].clone()
    side, junk = torch.cuda.Stream(), torch.full((3600,), 7.0, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    with torch.cuda.stream(side):
        sc.reset()
        sc.run(N, kernel=1)
        torch.cuda._sleep(20_000_000)                   # some ten milliseconds
        parts = [junk.clone() for _ in range(8)]        # written after the wait, then given back
        del parts
        got = sc.tally(0)[0]
        torch.cuda.synchronize()
    assert torch.allclose(got, want, rtol=1e-11, atol=1e-11)
    sc.close()
