"""Projections of dense event lists through angle and energy nodes (csrc/nodes.cu).

Against the FP64 oracle at the parity tolerances, and against the row kernel's
route (every line evaluated: energy classes off), whose FP32 sums it must
match to a few roundings (2e-6).  The sizes reach the edges of its tiles: 1 to
4 lines, voxel counts that end inside a run of 16 and a tile of 32, fewer than
32 scatter points, bin counts that are no multiple of the 8-row blocks, one
subset and as many subsets as angles, cells without events and cells of more
than one 256-event pass, streamed tables, the no-allocation call, events out
of range and events far from every line."""
from __future__ import annotations

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
import paper_2305_17111_gb300 as lm  # noqa: E402
from synthetic import preset, simulate  # noqa: E402

FWD_RTOL = 1e-5     # parity with the FP64 oracle
ROUTE_RTOL = 2e-6   # node route vs row route: FP32 sums in another order
IMG_RL2 = 1e-4

CASES = [
    ("tiny_8", {}, 3000),
    ("small_16", {}, 4000),
    ("small_16", {"line_keV": (140.0,), "yields": (1.0,), "windows": ((90.0, 160.0),)}, 3000),
    ("small_24", {"line_keV": (82.0, 154.0), "yields": (0.7, 0.3)}, 3000),
    ("small_24", {"line_keV": (82.0, 154.0, 270.0, 300.0), "yields": (0.4, 0.2, 0.2, 0.2),
                  "n_bins": 29, "n_angles": 7, "n_subsets": 7}, 3000),
    ("small_32_4w", {}, 6000),
    ("lmmew_32", {"n_bins": 37, "n_angles": 9, "n_subsets": 2, "scatter_n": 32}, 6000),
]


# the same models, and lists long enough for a reconstruction through the nodes
OSEM_CASES = [
    ("small_16", {}, 1_500_000),
    ("small_16", {"line_keV": (140.0,), "yields": (1.0,), "windows": ((90.0, 160.0),),
                  "n_subsets": 1}, 1_500_000),
    ("small_24", {"line_keV": (82.0, 154.0), "yields": (0.7, 0.3)}, 150_000),
    ("small_24", {"line_keV": (82.0, 154.0, 270.0, 300.0), "yields": (0.4, 0.2, 0.2, 0.2),
                  "n_bins": 29, "n_angles": 7, "n_subsets": 7}, 200_000),
    ("small_32_4w", {}, 250_000),
    ("lmmew_32", {"n_bins": 37, "n_angles": 9, "n_subsets": 2, "scatter_n": 32}, 60_000),
]


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


def _case(name, over, n_events, seed=3):
    sc = preset(name).with_(**over)
    ph = sc.make_phantom()
    ev = simulate(sc, n_events=n_events, seed=seed)
    rng = np.random.default_rng(seed)
    lam = (rng.uniform(0.2, 3.0, ph.rho.size) * (ph.rho.reshape(-1) > 0)).astype(np.float32)
    wt = rng.uniform(0.1, 1.0, len(ev)).astype(np.float32)
    gpu = lm.Model.from_scenario(sc, ph.rho)
    return sc, ph, ev, lam, wt, gpu, lm.DeviceEvents.from_list(ev)


def _repeat(ev, n, seed=9):
    """n events drawn from a list with replacement."""
    return ev.subset(np.random.default_rng(seed).integers(0, len(ev), size=n))


def _paths(gpu):
    """Path weights one projection of the node route visits."""
    return gpu.n_lines * gpu.nq * gpu.np_scatter


@pytest.mark.parametrize("name,over,n", CASES)
def test_projections_match_rows_and_oracle(name, over, n):
    sc, ph, ev, lam, wt, gpu, dev = _case(name, over, n)
    x, wv = torch.from_numpy(lam).cuda(), torch.from_numpy(wt).cuda()
    gpu.profile_enable(True)
    y = gpu.forward(dev, x)
    assert gpu.profile_read()["terms"] == _paths(gpu)      # the node route ran
    bp = gpu.backproject(dev, wv)
    assert gpu.profile_read()["terms"] == _paths(gpu)
    gpu.profile_enable(False)
    out = torch.empty_like(y)
    gpu.forward_noalloc(dev, x, out)
    assert torch.equal(out, y)
    gpu.set_energy_pruning(False)
    y_rows, bp_rows = gpu.forward(dev, x).double(), gpu.backproject(dev, wv).double()
    gpu.set_energy_pruning(True)
    assert float(((y.double() - y_rows) / y_rows).abs().max()) < ROUTE_RTOL
    on = bp_rows != 0
    assert bool((bp[~on] == 0).all())
    assert float(((bp.double() - bp_rows)[on] / bp_rows[on]).abs().max()) < ROUTE_RTOL
    idx = np.arange(0, len(ev), 13)
    ref = oracle.Model.from_scenario(sc, ph.rho).forward(ev.subset(idx), lam.astype(np.float64))
    got = y.cpu().numpy().astype(np.float64)[idx]
    assert float((np.abs(got - ref) / ref).max()) < FWD_RTOL
    gpu.close()


@pytest.mark.parametrize("name", ["tiny_8", "small_24"])
@pytest.mark.parametrize("less", [0, 1])
def test_either_side_of_two_events_per_angle(name, less):
    n = 2 * preset(name).n_angles - less
    sc, ph, ev, lam, wt, gpu, dev = _case(name, {}, n)
    x, wv = torch.from_numpy(lam).cuda(), torch.from_numpy(wt).cuda()
    gpu.profile_enable(True)
    y = gpu.forward(dev, x)
    assert (gpu.profile_read()["terms"] == _paths(gpu)) == (less == 0)
    gpu.profile_enable(False)
    bp = gpu.backproject(dev, wv).double()
    out = torch.empty_like(y)
    gpu.forward_noalloc(dev, x, out)
    assert torch.equal(out, y)
    gpu.set_energy_pruning(False)
    y_rows, bp_rows = gpu.forward(dev, x).double(), gpu.backproject(dev, wv).double()
    assert float(((y.double() - y_rows) / y_rows).abs().max()) < ROUTE_RTOL
    on = bp_rows != 0
    assert bool((bp[~on] == 0).all())
    assert float(((bp - bp_rows)[on] / bp_rows[on]).abs().max()) < ROUTE_RTOL
    gpu.close()


@pytest.mark.parametrize("name,over,n", OSEM_CASES)
def test_reconstruction_matches_the_row_route_and_resumes(name, over, n):
    sc, ph, ev, lam, wt, gpu, dev = _case(name, over, 4000, seed=5)
    dev = lm.DeviceEvents.from_list(_repeat(ev, n))
    n_sub = sc.n_subsets
    lam0 = torch.from_numpy((ph.rho.reshape(-1) > 0).astype(np.float32)).cuda()
    a, la = lam0.clone(), torch.zeros(2 * n_sub, dtype=torch.float64, device="cuda")
    gpu.osem(dev, a, n_sub, 2, loglik=la)
    assert not gpu.batch_tuning()["tuned"]                  # no row launch was tuned
    b = lam0.clone()
    gpu.osem(dev, b, n_sub, 2, 0, 0)
    assert torch.equal(a, b)                                # deterministic, with and without loglik
    c = lam0.clone()
    gpu.osem(dev, c, n_sub, 1)
    gpu.osem(dev, c, n_sub, 2, 1, 0)
    assert torch.equal(a, c)                                # resumed
    gpu.set_energy_pruning(False)
    d, ld = lam0.clone(), torch.zeros_like(la)
    gpu.osem(dev, d, n_sub, 2, loglik=ld)
    assert float((a - d).double().norm() / d.double().norm()) < ROUTE_RTOL
    assert float(((la - ld) / ld).abs().max()) < 1e-7
    gpu.close()


def test_streamed_tables_give_the_same_bits():
    sc, ph, ev, lam, wt, gpu, dev = _case("lmmew_32", {"n_angles": 10, "scatter_n": 32}, 5000)
    dense = lm.DeviceEvents.from_list(_repeat(ev, 120_000))
    x, wv = torch.from_numpy(lam).cuda(), torch.from_numpy(wt).cuda()
    lam0 = torch.from_numpy((ph.rho.reshape(-1) > 0).astype(np.float32)).cuda()
    img = lam0.clone()
    y, bp = gpu.forward(dev, x), gpu.backproject(dev, wv)
    gpu.osem(dense, img, 4, 2)
    assert not gpu.batch_tuning()["tuned"]
    for slots in (1, 3):
        gpu.set_table_streaming(slots)
        assert torch.equal(gpu.forward(dev, x), y)
        assert torch.equal(gpu.backproject(dev, wv), bp)
        img2 = lam0.clone()
        gpu.osem(dense, img2, 4, 2)
        assert torch.equal(img2, img)
    gpu.close()


def test_uneven_cells_and_bad_events():
    """All events in two cells (one of 3 000, several 256-event passes), with
    events out of range among them: those get NaN and are reported, the rest
    is what it is without them."""
    sc, ph, ev, lam, wt, gpu, dev = _case("small_24", {}, 10)
    rng = np.random.default_rng(8)
    n = 3300
    ang, bins = np.full(n, 3), np.where(np.arange(n) < 3000, 11, 12)
    e = rng.uniform(60.0, 290.0, n)
    x = torch.from_numpy(lam).cuda()
    good = lm.DeviceEvents(ang, bins, e)
    y = gpu.forward(good, x)
    w = torch.from_numpy(rng.uniform(0.5, 1.0, n).astype(np.float32)).cuda()
    bp = gpu.backproject(good, w)
    ang2, e2 = ang.copy(), e.copy()
    ang2[5], e2[3100] = sc.n_angles, 20.0
    bad = lm.DeviceEvents(ang2, bins, e2)
    y2 = gpu.forward(bad, x, check=False)
    with pytest.raises(lm.LmmewError, match="OUT_OF_RANGE"):
        gpu.check()
    assert bool(torch.isnan(y2[[5, 3100]]).all())
    keep = torch.ones(n, dtype=torch.bool, device="cuda")
    keep[[5, 3100]] = False
    assert torch.equal(y2[keep], y[keep])
    w0 = torch.where(keep, w, torch.zeros_like(w))
    bp2 = gpu.backproject(bad, w, check=False)
    with pytest.raises(lm.LmmewError, match="OUT_OF_RANGE"):
        gpu.check()
    ref = gpu.backproject(good, w0)
    assert float((bp2 - ref).double().norm() / ref.double().norm()) < ROUTE_RTOL
    gpu.set_energy_pruning(False)
    bp_rows = gpu.backproject(good, w).double()
    assert float((bp.double() - bp_rows).norm() / bp_rows.norm()) < ROUTE_RTOL
    gpu.close()


def test_energies_far_from_every_line():
    """A single 140 keV line in a wide window: events up to the reach of its
    scatter (8 sigma) follow the rows at 1e-4 of a value that is e^-32 of the
    peak there, events beyond carry the unscattered part alone, as the rows do."""
    sc, ph, ev, lam, wt, gpu, dev = _case("small_16", {"line_keV": (140.0,), "yields": (1.0,),
                                                       "windows": ((40.0, 300.0),)}, 10)
    n = 2000
    e = np.linspace(45.0, 230.0, n).astype(np.float32)
    rng = np.random.default_rng(1)
    evs = lm.DeviceEvents(rng.integers(0, sc.n_angles, n), rng.integers(8, 12, n), e)
    x = torch.from_numpy(lam).cuda()
    y = gpu.forward(evs, x).double().cpu().numpy()
    gpu.set_tile_events(64)
    small = 2 * sc.n_angles - 1      # the row route, with energy classes
    rows = np.concatenate([gpu.forward(lm.DeviceEvents(evs.angle[i:i + small], evs.bin[i:i + small],
                                                       evs.energy[i:i + small]), x).double().cpu().numpy()
                           for i in range(0, n, small)])
    on = rows > 0
    assert np.all(y[~on] == 0)
    rel = np.abs(y[on] - rows[on]) / rows[on]
    sigma = 0.1 * np.sqrt(140.0 * e[on]) / 2.3548
    back = 140.0 / (1.0 + 2.0 * 140.0 / 510.99895)
    out = np.maximum(np.maximum(e[on] - 140.0, back - e[on]), 0.0) / sigma
    assert rel[out < 4].max() < ROUTE_RTOL
    assert rel.max() < 1e-4
    gpu.close()


def test_batch_of_dense_and_sparse_realisations():
    """Dense realisations run through the nodes, sparse ones share row launches;
    each equals its own lm_osem bit for bit, and a bad event is refused."""
    sc, ph, ev, lam, wt, gpu, dev = _case("small_24", {}, 4000)
    sizes = [150_000, 300, 0, 200_000, 1500]
    evs = [_repeat(ev, n, seed=60 + i) for i, n in enumerate(sizes)]
    devs = [lm.DeviceEvents.from_list(e) for e in evs]
    rng = np.random.default_rng(0)
    lam0 = torch.from_numpy(np.stack([rng.uniform(0.5, 2.0, ph.rho.size) * (ph.rho.reshape(-1) > 0)
                                      for _ in sizes]).astype(np.float32)).cuda()
    n_sub, n_it = sc.n_subsets, 2
    imgs, ll = lam0.clone(), torch.zeros(len(sizes), n_it * n_sub, dtype=torch.float64, device="cuda")
    gpu.osem_batch(devs, imgs, n_sub, n_it, loglik=ll)
    for i, d in enumerate(devs):
        one, l1 = lam0[i].clone(), torch.zeros(n_it * n_sub, dtype=torch.float64, device="cuda")
        gpu.osem(d, one, n_sub, n_it, loglik=l1)
        assert torch.equal(imgs[i], one), f"realisation {i}"
        assert torch.equal(ll[i], l1), f"realisation {i}"
    bad = evs[3].subset(np.arange(len(evs[3])))
    bad.energy[7] = 5.0
    devs[3] = lm.DeviceEvents.from_list(bad)
    before = imgs.clone()
    with pytest.raises(lm.LmmewError, match="OUT_OF_RANGE"):
        gpu.osem_batch(devs, imgs, n_sub, n_it)
    assert torch.equal(imgs, before)
    gpu.close()
