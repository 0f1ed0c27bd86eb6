"""The warp pools at the edges of their steps: fewer histories than lanes, one
step's worth, a pool's worth and one more, blocks of one warp to eight.  FP64,
against the history kernel: every history has its own random numbers, so the
counters agree exactly and the tallies to the rounding of their sums (at most
a few thousand FP64 additions of like sign: 1e-12)."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


def _run(desc, n, kernel, block, grad=False):
    from paper_2304_06226_gb300.engine import Scene
    sc = Scene(desc)
    sc.run(n, kernel=kernel, block_size=block, want_grad=grad, secondaries=2 if grad else 0)
    torch.cuda.synchronize()
    raw = [sc.raw(q) for q in range(sc.n_inst)]
    cnt = sc.counters()
    sc.close()
    return cnt, {k: np.stack([r[k] for r in raw]) for k in ("sum", "sumsq", "J")}


SCENES = {"powder": lambda: W.powder(precision="f64", g=(0.5, 2.0, 2.0)), "guide": lambda: W.guide(precision="f64"),
          "slab": lambda: W.slab(g=3.0), "chopper": lambda: W.chopper(precision="f64"),
          "batched": lambda: W.batched(n_instances=3, precision="f64"),
          "imaging": lambda: W.imaging(n_prims=60, precision="f64", psd_bins=16)}


@pytest.mark.parametrize("block", [32, 160, 256])
@pytest.mark.parametrize("n", [1, 31, 32, 33, 64, 65, 4097])
@pytest.mark.parametrize("scene", sorted(SCENES))
def test_pool_steps(scene, n, block):
    desc = SCENES[scene]()
    grad = scene in ("batched", "imaging")
    cnt, got = _run(desc, n, 3, block, grad)
    ref_cnt, ref = _run(desc, n, 1, 128, grad)
    assert cnt == ref_cnt
    for k, v in ref.items():
        if v.size:
            assert np.allclose(got[k], v, rtol=1e-12, atol=1e-12 * max(1e-300, np.abs(v).max())), k


@pytest.mark.parametrize("precision", ["f32", "f64"])
@pytest.mark.parametrize("scene", ["slab", "guide"])
def test_every_history_runs_once_and_as_in_the_history_kernel(scene, precision):
    """Slots return to the stacks a step popped them from.  A slot listed twice or
    lost would end a history early, twice or never: each path is that of the
    history kernel, word for word (the geometry is explicit arithmetic); the
    weight, a product of at most a hundred factors, to their rounding."""
    from paper_2304_06226_gb300.engine import Scene, new_records, records_to_numpy
    n, out = 100_003, []
    sc = Scene({"slab": lambda: W.slab(g=3.0, precision=precision), "guide": lambda: W.guide(precision=precision)}[scene]())
    for kernel in (1, 3):
        rec = new_records(n)
        sc.run(n, kernel=kernel, records=rec)
        torch.cuda.synchronize()
        out.append(records_to_numpy(rec))
    sc.close()
    for k, v in out[0].items():
        if k == "w_final":
            assert np.allclose(out[1][k], v, rtol=100 * (2.0 ** -23 if precision == "f32" else 2.0 ** -52), atol=0.0)
        else:
            assert np.array_equal(out[1][k], v, equal_nan=v.dtype.kind == "f"), k


# Scenes whose weights stay 1: the pools count in shared memory, the event
# kernel adds w and w^2 with FP64 atomics; both are whole numbers and equal.
# 4096 bins are the most a histogram holds; with one more the pools add weights.
UNIT = {"powder": lambda p: W.powder(precision=p), "powder_4096": lambda p: W.powder(precision=p, nbins=4096),
        "powder_4097": lambda p: W.powder(precision=p, nbins=4097),
        "orders": lambda p: W.total_scattering(precision=p, g=1.0),
        "chopper": lambda p: W.chopper(precision=p), "slit": lambda p: W.moderator_test(precision=p, temperature=300.0),
        "slab": lambda p: W.slab(g=1.0, precision=p)}


@pytest.mark.parametrize("n", [1, 100, 50_001])
@pytest.mark.parametrize("precision", ["f32", "f64"])
@pytest.mark.parametrize("scene", sorted(UNIT))
def test_counting_equals_summing(scene, precision, n):
    desc = UNIT[scene](precision)
    cnt, got = _run(desc, n, 3, 256)
    ref_cnt, ref = _run(desc, n, 2, 256)
    assert cnt == ref_cnt
    assert (got["sum"] == ref["sum"]).all() and (got["sumsq"] == ref["sumsq"]).all()
    assert (got["sum"] == np.rint(got["sum"])).all() and (got["sum"] == got["sumsq"]).all()


def test_counting_adds_to_what_is_there_and_stops_with_a_bias():
    from paper_2304_06226_gb300.engine import Scene
    sc = Scene(W.powder())
    sc.run(1000, kernel=3, first=0)
    sc.run(1000, kernel=3, first=1000)
    two = sc.raw()["sum"].copy()
    sc.reset()
    sc.run(2000, kernel=3)
    assert (sc.raw()["sum"] == two).all()
    sc.reset()
    sc.set_bias(0, (1.0, 2.0, 1.0))   # weights now differ from 1
    sc.run(20_000, kernel=3)
    raw = sc.raw()
    sc.close()
    assert not (raw["sum"] == raw["sumsq"]).all()


def _counting(desc, n=1000, **kw):
    from paper_2304_06226_gb300.engine import Scene
    sc = Scene(desc)
    sc.run(n, kernel=3, **kw)
    torch.cuda.synchronize()
    form = sc.launch_counting()
    sc.close()
    return form


@pytest.mark.parametrize("precision", ["f32", "f64"])
def test_which_scenes_count(precision):
    assert all(_counting(UNIT[k](precision)) for k in UNIT if k != "powder_4097")
    assert not _counting(UNIT["powder_4097"](precision))
    assert not _counting(W.guide(precision=precision))                      # mirrors
    assert not _counting(W.slab(g=3.0, precision=precision))                # a bias
    assert not _counting(W.imaging(n_prims=60, precision=precision, psd_bins=16))   # a grid
    grad = W.imaging(n_prims=10, precision=precision, psd_bins=16)          # no grid, no bias
    grad["bias"][:] = 1.0
    assert _counting(grad) and not _counting(grad, want_grad=True)


@pytest.mark.parametrize("cap,form", [(1 << 21, True), ((1 << 21) + 1, False), (2**31 - 1, False)])
def test_counting_stops_above_the_event_cap_its_bound_is_for(cap, form):
    """A count stays below 2^32 while no history has more events than this."""
    desc = W.powder()
    desc["event_cap"] = cap
    assert _counting(desc) is form


def test_a_bias_set_later_ends_counting_and_none_brings_it_back():
    from paper_2304_06226_gb300.engine import Scene
    sc, seen = Scene(W.powder()), []
    for g in (1.0, 2.0, 1.0):
        sc.set_bias(0, (1.0, g, 1.0))
        sc.run(1000, kernel=3)
        seen.append(sc.launch_counting())
    sc.close()
    assert seen == [True, False, True]


@pytest.mark.parametrize("block", [32, 160, 256])
@pytest.mark.parametrize("precision", ["f32", "f64"])
@pytest.mark.parametrize("scene", ["powder_4096", "orders", "chopper", "slab"])
def test_histogram_emptied_while_the_block_scores(scene, precision, block):
    """Every warp empties its block's histogram many times while the others score
    (the flag's 64 crossings instead of 2^23): no count is lost or added twice."""
    from paper_2304_06226_gb300 import native as N
    from paper_2304_06226_gb300.engine import Scene
    n = 1_000_001
    desc = UNIT[scene](precision)
    sc = Scene(desc)
    sc.set_test_flags(N.TP_TEST_SMALL_HIST_INTERVAL)
    sc.run(n, kernel=3, block_size=block, ctas_per_sm=1)
    torch.cuda.synchronize()
    assert sc.launch_counting()
    got, cnt = sc.raw(), sc.counters()
    assert cnt["crossings"] > 10 * 64 * 152 * (block // 32)   # ten times a warp and more
    sc.close()
    ref_cnt, ref = _run(desc, n, 2, 256)
    assert cnt == ref_cnt
    assert (got["sum"] == ref["sum"][0]).all() and (got["sumsq"] == ref["sumsq"][0]).all()


@pytest.mark.parametrize("block,ctas", [(32, 1), (160, 0), (256, 0)])
@pytest.mark.parametrize("n", [151, 609, 3001, 19_457, 20_011, 130_003])
@pytest.mark.parametrize("scene,precision", [("slab", "f64"), ("chopper", "f64"), ("imaging", "f64"), ("imaging", "f32")])
def test_every_history_is_claimed_once_whatever_the_share(scene, precision, n, block, ctas):
    """Runs that end within the histories the warps start with, at their edge (19456 =
    152 * 4 * 32 full warps) and beyond it; FP32 shares of a grid scene."""
    from paper_2304_06226_gb300.engine import Scene
    desc = {"slab": lambda: W.slab(g=3.0), "chopper": lambda: W.chopper(precision="f64"),
            "imaging": lambda: W.imaging(n_prims=60, precision=precision, psd_bins=16)}[scene]()
    seen = []
    sc = Scene(desc)
    for kernel in (1, 3):
        sc.reset()
        sc.run(n, kernel=kernel, block_size=block, ctas_per_sm=ctas)
        torch.cuda.synchronize()
        seen.append((sc.counters(), sc.raw()["sum"]))
    sc.close()
    assert seen[0][0] == seen[1][0] and seen[0][0]["histories"] == n
    tol = 1e-12 if precision == "f64" else 1e-5   # (FP32: a group of up to 32 weights is summed in FP32)
    assert np.allclose(seen[1][1], seen[0][1], rtol=tol, atol=tol * seen[0][1].max())
