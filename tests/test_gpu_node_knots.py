"""Attenuation knots inside the scattered energies (csrc/nodes.cu): mu(E') has a
kink there, which the direction nodes may not smooth over.  Images of one hot
voxel, few scatter points and long ways through water leave nothing to average
the kink away; energies go over the whole window.  Forward projections and back
projections of single events against the FP64 oracle; the collimator is wide
enough that no scatter point falls below its floor, which the oracle has not.

Tolerance: exponents of up to 9 bits with two FP32 roundings (1.1e-6), some ten
products (6e-7) and the interpolation (2e-8), twice: 4e-6, wherever a value is
above 1e-3 of the largest of its (angle, bin), or of its event's row."""
from __future__ import annotations

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
import paper_2305_17111_gb300 as lm  # noqa: E402
from synthetic import preset  # noqa: E402
from synthetic.mc import EventList  # noqa: E402

RTOL = 4e-6
MANY = dict(knot_keV=(60.0, 75.0, 100.0, 131.5, 154.0, 156.0, 200.0, 269.9, 300.0),
            mu_water_cm=(0.21, 0.19, 0.172, 0.155, 0.15, 0.147, 0.135, 0.12, 0.119))
WATER = dict(n=16, pixel_cm=2.5, scatter_n=2, n_angles=12, n_bins=20)   # 40 cm, 4 scatter points
WIDE = dict(coll_fwhm0_cm=30.0, coll_fwhm_slope=0.0)
CASES = [
    ("lmmew_32", {}, False),
    ("small_16", WATER, True),
    ("small_16", {**WATER, **MANY}, True),
    ("small_16", {**MANY, "line_keV": (82.0, 154.0, 270.0, 300.0), "yields": (0.4, 0.2, 0.2, 0.2),
                  "n_angles": 7, "n_subsets": 1}, False),
]


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


def _model(name, over, water):
    sc = preset(name).with_(**over, **WIDE)
    rho = np.ones((sc.n, sc.n), np.float32) if water else sc.make_phantom().rho
    return sc, rho, lm.Model.from_scenario(sc, rho)


def _list(a, b, e):
    z = np.zeros(a.size, np.int32)
    return EventList(a.astype(np.uint16), b.astype(np.uint16), e.astype(np.float32), z,
                     z.astype(np.uint8), z.astype(bool))


@pytest.mark.parametrize("name,over,water", CASES)
def test_one_voxel_forward_matches_the_oracle(name, over, water):
    sc, rho, gpu = _model(name, over, water)
    angles, bins = np.arange(0, sc.n_angles, 3), np.arange(1, sc.n_bins, 3)
    per = 40
    rng = np.random.default_rng(1)
    a, b = np.meshgrid(angles, bins, indexing="ij")
    a, b = np.repeat(a.reshape(-1), per), np.repeat(b.reshape(-1), per)
    e = np.tile(np.linspace(61.0, 284.0, per), a.size // per) + rng.uniform(-2.5, 2.5, a.size)
    ev = _list(a, b, e)
    dev, orc = lm.DeviceEvents.from_list(ev), oracle.Model.from_scenario(sc, rho)
    voxels = np.flatnonzero(rho.reshape(-1) > 0)
    for q in voxels[[len(voxels) // 7, len(voxels) // 2]]:
        lam = np.zeros(sc.n * sc.n)
        lam[q] = 2.0
        gpu.profile_enable(True)
        y = gpu.forward(dev, torch.from_numpy(lam.astype(np.float32)).cuda())
        assert gpu.profile_read()["terms"] == gpu.n_lines * gpu.nq * gpu.np_scatter   # the node route
        gpu.profile_enable(False)
        y = y.double().cpu().numpy().reshape(-1, per)
        ref = orc.forward(ev, lam).reshape(-1, per)
        on = (ref > 1e-3 * ref.max(axis=1, keepdims=True)) & (ref > 1e-25)
        assert on.sum() > 200
        assert float((np.abs(y - ref)[on] / ref[on]).max()) < RTOL
    gpu.close()


def test_narrow_collimator_at_the_parity_tolerance():
    """The 32 x 32 scanner as it is: bins that see few paths.  The collimator's
    floor drops points there, so the bound is the parity tolerance, above 1 % of
    each (angle, bin)'s largest value."""
    sc = preset("lmmew_32")
    rho = sc.make_phantom().rho
    gpu, orc = lm.Model.from_scenario(sc, rho), oracle.Model.from_scenario(sc, rho)
    per = 40
    a, b = np.meshgrid(np.arange(0, 32, 3), np.arange(1, 32, 3), indexing="ij")
    a, b = np.repeat(a.reshape(-1), per), np.repeat(b.reshape(-1), per)
    rng = np.random.default_rng(1)
    ev = _list(a, b, np.tile(np.linspace(61.0, 284.0, per), a.size // per) + rng.uniform(-2.5, 2.5, a.size))
    dev = lm.DeviceEvents.from_list(ev)
    voxels = np.flatnonzero(rho.reshape(-1) > 0)
    for q in voxels[[len(voxels) // 7, len(voxels) // 2]]:
        lam = np.zeros(1024)
        lam[q] = 2.0
        y = gpu.forward(dev, torch.from_numpy(lam.astype(np.float32)).cuda()).double().cpu().numpy()
        ref = orc.forward(ev, lam)
        on = ref > 1e-2 * ref.reshape(-1, per).max(axis=1).repeat(per)
        assert float((np.abs(y - ref)[on] / ref[on]).max()) < 1e-5
    gpu.close()


@pytest.mark.parametrize("name,over,water", CASES)
def test_single_events_back_match_the_oracle(name, over, water):
    sc, rho, gpu = _model(name, over, water)
    orc = oracle.Model.from_scenario(sc, rho)
    n = 12 * sc.n_angles
    rng = np.random.default_rng(2)
    a, b = rng.integers(0, sc.n_angles, n), rng.integers(0, sc.n_bins, n)
    ev = _list(a, b, rng.uniform(62.0, 280.0, n))
    dev = lm.DeviceEvents.from_list(ev)
    for j in rng.integers(0, n, 12):
        w = torch.zeros(n, device="cuda")
        w[int(j)] = 1.5
        gpu.profile_enable(True)
        bp = gpu.backproject(dev, w).double().cpu().numpy()
        assert gpu.profile_read()["terms"] == gpu.n_lines * gpu.nq * gpu.np_scatter
        gpu.profile_enable(False)
        ref = 1.5 * orc.row_image(a[j], b[j], float(ev.energy[j]))
        on = ref > 1e-3 * ref.max()
        assert float((np.abs(bp - ref)[on] / ref[on]).max()) < RTOL
    gpu.close()
