"""Set-up of a scatter grid with more points than the point order stages at a
time (1024, csrc/setup.cu) and a bin count that ends inside a collimator
thread's run of 8: sensitivities and projections against the FP64 oracle at
the parity tolerances, on the rows' route, which reads every table."""
from __future__ import annotations

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
import paper_2305_17111_gb300 as lm  # noqa: E402
from synthetic import preset, simulate  # noqa: E402

FWD_RTOL = 1e-5
SENS_RTOL = 2e-6   # FP64 sums of terms whose window masses are FP32


@pytest.mark.parametrize("n,pixel_cm,n_bins", [(80, 0.4, 45), (64, 0.5, 71)])
def test_set_up_beyond_one_stage_of_points(n, pixel_cm, n_bins):
    sc = preset("lmmew_64").with_(n=n, pixel_cm=pixel_cm, n_angles=3, n_bins=n_bins, scatter_n=n,
                                  n_subsets=3)
    ph = sc.make_phantom()
    assert int((ph.rho > 0).sum()) > 1024
    orc = oracle.Model.from_scenario(sc, ph.rho)
    gpu = lm.Model.from_scenario(sc, ph.rho)
    for s in (0, 2, -1):
        np.testing.assert_allclose(gpu.sensitivity(s).cpu().numpy(), orc.sensitivity(s, sc.n_subsets),
                                   rtol=SENS_RTOL, atol=0)
    ev = simulate(sc, n_events=18, seed=3)          # too few for the energy nodes
    lam = (np.random.default_rng(3).uniform(0.2, 3.0, ph.rho.size) * (ph.rho.reshape(-1) > 0))
    lam = lam.astype(np.float32)
    got = gpu.forward(lm.DeviceEvents.from_list(ev), torch.from_numpy(lam).cuda())
    ref = orc.forward(ev, lam.astype(np.float64))
    rel = np.abs(got.cpu().numpy().astype(np.float64) - ref) / np.abs(ref)
    assert float(rel.max()) < FWD_RTOL
    gpu.close()
