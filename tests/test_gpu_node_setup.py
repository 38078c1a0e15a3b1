"""Set-up of the node route's tables (csrc/nodes.cu): the paths of a scatter
point are sorted in shared memory up to 16 384 voxels and by the global sort
above, so projections through the nodes are compared with the rows' (the same
model, FP32 sums in another order) at voxel counts on either side of that and
of the sort's powers of two; and what the tables add to the creation of a
small model."""
from __future__ import annotations

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
import paper_2305_17111_gb300 as lm  # noqa: E402
from synthetic import preset  # noqa: E402
from synthetic.mc import EventList  # noqa: E402

ROUTE_RTOL = 2e-6   # node route vs row route: FP32 sums in another order
PARITY_RTOL = 1e-5  # parity with the FP64 oracle


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


def _events(sc, per_cell, seed):
    """per_cell events in every (angle, bin) cell, energies over the lines' scatter."""
    rng = np.random.default_rng(seed)
    a, b = np.meshgrid(np.arange(sc.n_angles), np.arange(sc.n_bins), indexing="ij")
    a, b = np.repeat(a.reshape(-1), per_cell), np.repeat(b.reshape(-1), per_cell)
    return lm.DeviceEvents(a, b, rng.uniform(62.0, 280.0, a.size).astype(np.float32))


# pixels, scatter cells, voxels of the support (the first ones): 64 and 65 (the
# smallest sort and past it), a power of two, the largest sort in shared memory
@pytest.mark.parametrize("n,scatter_n,voxels", [(8, 4, 64), (9, 3, 65), (32, 8, 1024), (128, 4, 16384)])
def test_projections_for_every_sort_size(n, scatter_n, voxels):
    sc = preset("tiny_8").with_(n=n, pixel_cm=25.6 / n, n_bins=9, scatter_n=scatter_n)
    rho = np.ones((n, n), np.float32)
    support = (np.arange(n * n) < voxels).astype(np.uint8)
    gpu = lm.Model.from_scenario(sc, rho, support=support)
    assert gpu.nq == voxels
    dev = _events(sc, 5, n)
    rng = np.random.default_rng(voxels)
    x = torch.from_numpy((rng.uniform(0.2, 3.0, n * n) * support).astype(np.float32)).cuda()
    wv = torch.from_numpy(rng.uniform(0.1, 1.0, len(dev)).astype(np.float32)).cuda()
    gpu.profile_enable(True)
    y = gpu.forward(dev, x).double()
    assert gpu.profile_read()["terms"] == gpu.n_lines * gpu.nq * gpu.np_scatter    # the node route
    gpu.profile_enable(False)
    bp = gpu.backproject(dev, wv).double()
    gpu.set_energy_pruning(False)
    y_rows, bp_rows = gpu.forward(dev, x).double(), gpu.backproject(dev, wv).double()
    assert float(((y - y_rows) / y_rows).abs().max()) < ROUTE_RTOL
    on = bp_rows != 0
    assert bool((bp[~on] == 0).all())
    assert float(((bp - bp_rows)[on] / bp_rows[on]).abs().max()) < ROUTE_RTOL
    gpu.close()


@pytest.mark.parametrize("voxels", [16385, 16641])
def test_global_sort_matches_the_oracle(voxels):
    """Past the largest sort in shared memory.  Nine scatter points: the rows'
    rounding of a single path (5e-6) is too coarse a reference there."""
    sc = preset("tiny_8").with_(n=129, pixel_cm=25.6 / 129, n_bins=9, scatter_n=3)
    rho = np.ones((129, 129), np.float32)
    support = (np.arange(129 * 129) < voxels).astype(np.uint8)
    gpu = lm.Model.from_scenario(sc, rho, support=support)
    orc = oracle.Model.from_scenario(sc, rho, support=support)
    assert gpu.nq == voxels
    dev = _events(sc, 5, 129)
    z = np.zeros(len(dev), np.int32)
    ev = EventList(dev.angle.cpu().numpy().astype(np.uint16), dev.bin.cpu().numpy().astype(np.uint16),
                   dev.energy.cpu().numpy(), z, z.astype(np.uint8), z.astype(bool))
    rng = np.random.default_rng(voxels)
    lam = (rng.uniform(0.2, 3.0, 129 * 129) * support).astype(np.float32)
    w = rng.uniform(0.1, 1.0, len(dev)).astype(np.float32)
    gpu.profile_enable(True)
    y = gpu.forward(dev, torch.from_numpy(lam).cuda()).double().cpu().numpy()
    assert gpu.profile_read()["terms"] == gpu.n_lines * gpu.nq * gpu.np_scatter    # the node route
    ref = orc.forward(ev, lam.astype(np.float64))
    assert float((np.abs(y - ref) / ref).max()) < PARITY_RTOL
    bp = gpu.backproject(dev, torch.from_numpy(w).cuda()).double().cpu().numpy()
    ref = orc.backproject(ev, w)
    on = ref > 0
    assert np.all(bp[~on] == 0)
    assert float((np.abs(bp - ref)[on] / ref[on]).max()) < PARITY_RTOL
    gpu.close()


def test_tables_of_a_small_model_take_few_launches():
    """Nine kernels; the same model at a resolution whose energy nodes are too
    many for the route has none of them."""
    sc = preset("small_24").with_(n_angles=24, scatter_n=12)
    rho = sc.make_phantom().rho
    count = {}
    for frac in (0.10, 0.02):
        gpu = lm.Model.from_scenario(sc.with_(fwhm_frac=frac), rho)
        count[frac] = gpu.profile_read()["kernels"]
        gpu.close()
    assert 1 <= count[0.10] - count[0.02] <= 9


def test_node_tables_are_part_of_the_accounts():
    """lm_model_info's table bytes and set-up time cover the node tables: 12 + 4
    bytes a line for every pair of voxel and scatter point at least."""
    sc = preset("small_24").with_(n_angles=24, scatter_n=12)
    rho = sc.make_phantom().rho
    ms = {}
    for frac in (0.10, 0.02):
        for _ in range(12):
            gpu = lm.Model.from_scenario(sc.with_(fwhm_frac=frac), rho)
            ms[frac] = min(ms.get(frac, 1e9), gpu.setup_ms)
            nodes = gpu.table_bytes - gpu.table_streaming()[1]
            if frac == 0.10:
                assert nodes > (12 + 4 * gpu.n_lines) * gpu.nq * gpu.np_scatter
            else:
                assert nodes == 0
            gpu.close()
    assert ms[0.10] > ms[0.02] + 0.05
