"""Events far from every energy a scattered photon can have (csrc/nodes.cu): up to
8 sigma, where the reach ends, a value is e^-32 of the peak and the energy and
direction nodes have to carry its relative precision; OSEM divides by it.
Against the FP64 oracle, with a collimator wide enough that no scatter point
falls below its floor (which the oracle has not), over resolutions and lines
whose Gaussians bend differently over the stencils.

Tolerance 1e-5, the parity bar: interpolation 3e-6 at 8 sigma and FP32 terms
that weights of both signs amplify some three times (2e-6) leave a factor 2."""
from __future__ import annotations

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
import paper_2305_17111_gb300 as lm  # noqa: E402
from synthetic import preset  # noqa: E402
from synthetic.mc import EventList  # noqa: E402

RTOL = 1e-5
ME_C2 = 510.99895


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


@pytest.mark.parametrize("line,frac", [(140.0, 0.10), (82.0, 0.10), (270.0, 0.08), (60.0, 0.14)])
@pytest.mark.parametrize("one_voxel", [False, True])
def test_values_keep_their_precision_to_the_end_of_the_reach(line, frac, one_voxel):
    sc = preset("small_16").with_(line_keV=(line,), yields=(1.0,), windows=((1.0, 600.0),), fwhm_frac=frac,
                                  coll_fwhm0_cm=30.0, coll_fwhm_slope=0.0)
    rho = sc.make_phantom().rho
    gpu, orc = lm.Model.from_scenario(sc, rho), oracle.Model.from_scenario(sc, rho)
    back = line / (1.0 + 2.0 * line / ME_C2)
    sigma = lambda e: frac * np.sqrt(140.0 * e) / 2.3548  # noqa: E731
    lo, hi = back - 7.9 * sigma(back), line + 7.9 * sigma(line)
    e = np.linspace(max(lo, 2.0), hi, 600).astype(np.float32)
    rng = np.random.default_rng(5)
    z = np.zeros(e.size, np.int32)
    ev = EventList(rng.integers(0, sc.n_angles, e.size).astype(np.uint16),
                   rng.integers(0, sc.n_bins, e.size).astype(np.uint16), e, z, z.astype(np.uint8),
                   z.astype(bool))
    lam = rng.uniform(0.2, 3.0, rho.size) * (rho.reshape(-1) > 0)
    if one_voxel:
        on = np.flatnonzero(lam)
        lam[np.delete(on, on.size // 3)] = 0.0
    lam = lam.astype(np.float32)
    gpu.profile_enable(True)
    y = gpu.forward(lm.DeviceEvents.from_list(ev), torch.from_numpy(lam).cuda()).double().cpu().numpy()
    assert gpu.profile_read()["terms"] == gpu.nq * gpu.np_scatter        # the node route
    ref = orc.forward(ev, lam.astype(np.float64))
    on = ref > 1e-30
    assert on.sum() > 500
    assert float((np.abs(y - ref)[on] / ref[on]).max()) < RTOL
    gpu.close()
