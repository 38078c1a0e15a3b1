"""The row kernel in the projections that still take it: lists of fewer than 2
events per detector angle.  Scanners of 128 angles, so that 255 events, most of
them at one angle, fill tiles of 32, 64 and 128 events of a class and leave a
ragged one; 1 to 4 lines; energy pruning and streamed path tables; a scatter grid
finer than the point order's stage.  Against the FP64 oracle at the parity
tolerance, and bit for bit over tile sizes and table blocks.  Every call's route
is checked: the node route visits a fixed number of paths."""
from __future__ import annotations

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
import paper_2305_17111_gb300 as lm  # noqa: E402
from synthetic import preset  # noqa: E402
from synthetic.mc import EventList  # noqa: E402

RTOL = 1e-5        # parity with the FP64 oracle
PRUNE_RTOL = 2e-6  # rows with and without the lines out of reach: FP32 sums of other lengths


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


def _list(sc, n, crowd, seed):
    """n events, `crowd` of them at one angle in neighbouring bins."""
    rng = np.random.default_rng(seed)
    a, b = rng.integers(0, sc.n_angles, n), rng.integers(0, sc.n_bins, n)
    a[:crowd] = sc.n_angles // 3
    b[:crowd] = sc.n_bins // 2 + rng.integers(-2, 3, crowd)
    b[crowd:] = np.clip(b[crowd:], sc.n_bins // 4, 3 * sc.n_bins // 4)
    order, z = rng.permutation(n), np.zeros(n, np.int32)
    e = rng.uniform(62.0, min(1.02 * max(sc.line_keV), 299.0), n)
    return EventList(a[order].astype(np.uint16), b[order].astype(np.uint16), e.astype(np.float32), z,
                     z.astype(np.uint8), z.astype(bool))


def _case(name, over, n, crowd, seed=4):
    sc = preset(name).with_(**over)
    rho = sc.make_phantom().rho
    ev = _list(sc, n, crowd, seed)
    rng = np.random.default_rng(seed)
    lam = (rng.uniform(0.2, 3.0, rho.size) * (rho.reshape(-1) > 0)).astype(np.float32)
    w = rng.uniform(0.1, 1.0, n).astype(np.float32)
    return sc, rho, ev, lam, w, lm.Model.from_scenario(sc, rho), lm.DeviceEvents.from_list(ev)


def _rows(gpu, call):
    """The result and the terms of a call that has to go through the rows."""
    gpu.profile_enable(True)
    out = call().clone()
    terms = gpu.profile_read()["terms"]
    gpu.profile_enable(False)
    assert terms > 0 and terms != gpu.n_lines * gpu.nq * gpu.np_scatter
    return out, terms


@pytest.mark.parametrize("name,over", [
    ("small_24", {"n_angles": 128}),
    ("small_24", {"n_angles": 128, "line_keV": (140.0,), "yields": (1.0,)}),
    ("small_24", {"n_angles": 128, "line_keV": (82.0, 154.0), "yields": (0.7, 0.3), "n_bins": 29}),
    ("small_16", {"n_angles": 128, "line_keV": (82.0, 154.0, 270.0, 300.0), "yields": (0.4, 0.2, 0.2, 0.2)}),
    ("lmmew_32", {"n_angles": 128, "scatter_n": 32})])
@pytest.mark.parametrize("pruning", [True, False])
def test_rows_of_every_tile_size_match_the_oracle(name, over, pruning):
    sc, rho, ev, lam, w, gpu, dev = _case(name, over, 255, 230)
    gpu.set_energy_pruning(pruning)
    x, wv = torch.from_numpy(lam).cuda(), torch.from_numpy(w).cuda()
    got = {}
    for tile in (128, 64, 32):
        gpu.set_tile_events(tile)
        y, _ = _rows(gpu, lambda: gpu.forward(dev, x))
        bp, _ = _rows(gpu, lambda: gpu.backproject(dev, wv))
        out = torch.empty_like(y)
        gpu.forward_noalloc(dev, x, out)
        assert torch.equal(out, y)
        got[tile] = (y, bp)
    for tile in (64, 32):
        assert torch.equal(got[tile][0], got[128][0]) and torch.equal(got[tile][1], got[128][1])
    orc = oracle.Model.from_scenario(sc, rho)
    y, bp = (t.double().cpu().numpy() for t in got[32])
    ref = orc.forward(ev, lam.astype(np.float64))
    assert float((np.abs(y - ref) / ref).max()) < RTOL
    ref = orc.backproject(ev, w.astype(np.float64))
    on = ref > 0
    assert float((np.abs(bp - ref)[on] / ref[on]).max()) < RTOL
    gpu.close()


@pytest.mark.parametrize("tile", [32, 64, 128])
def test_pruned_rows_drop_only_lines_out_of_reach(tile):
    sc, rho, ev, lam, w, gpu, dev = _case("small_24", {"n_angles": 128}, 255, 200)
    gpu.set_tile_events(tile)
    x, wv = torch.from_numpy(lam).cuda(), torch.from_numpy(w).cuda()
    on = [_rows(gpu, lambda: gpu.forward(dev, x)), _rows(gpu, lambda: gpu.backproject(dev, wv))]
    gpu.set_energy_pruning(False)
    gpu.set_tile_events(tile)
    off = [_rows(gpu, lambda: gpu.forward(dev, x)), _rows(gpu, lambda: gpu.backproject(dev, wv))]
    for (a, terms_on), (b, terms_off) in zip(on, off):
        assert terms_on < terms_off
        m = b != 0
        assert bool((a[~m] == 0).all())
        assert float(((a - b)[m].double() / b[m].double()).abs().max()) < PRUNE_RTOL
    gpu.close()


@pytest.mark.parametrize("slots", [1, 3, 7])
def test_streamed_rows_match_resident_ones(slots):
    sc, rho, ev, lam, w, gpu, dev = _case("small_24", {"n_angles": 20}, 39, 20)
    x, wv = torch.from_numpy(lam).cuda(), torch.from_numpy(w).cuda()
    y, _ = _rows(gpu, lambda: gpu.forward(dev, x))
    bp, _ = _rows(gpu, lambda: gpu.backproject(dev, wv))
    gpu.set_table_streaming(slots)
    for _ in range(2):          # again: blocks resident from the last call
        assert torch.equal(_rows(gpu, lambda: gpu.forward(dev, x))[0], y)
        assert torch.equal(_rows(gpu, lambda: gpu.backproject(dev, wv))[0], bp)
    out = torch.empty_like(y)
    gpu.forward_noalloc(dev, x, out)
    assert torch.equal(out, y)
    ref = oracle.Model.from_scenario(sc, rho).forward(ev, lam.astype(np.float64))
    assert float((np.abs(y.double().cpu().numpy() - ref) / ref).max()) < RTOL
    gpu.close()


@pytest.mark.parametrize("n,pixel_cm,n_bins", [(80, 0.4, 45), (64, 0.5, 71)])
def test_rows_of_a_scatter_grid_beyond_one_stage(n, pixel_cm, n_bins):
    """More points than the point order stages at a time (1024)."""
    over = dict(n=n, pixel_cm=pixel_cm, n_angles=3, n_bins=n_bins, scatter_n=n, n_subsets=3)
    sc, rho, ev, lam, w, gpu, dev = _case("lmmew_64", over, 5, 2)
    assert gpu.np_scatter > 1024
    y, _ = _rows(gpu, lambda: gpu.forward(dev, torch.from_numpy(lam).cuda()))
    ref = oracle.Model.from_scenario(sc, rho).forward(ev, lam.astype(np.float64))
    assert float((np.abs(y.double().cpu().numpy() - ref) / ref).max()) < RTOL
    gpu.close()
