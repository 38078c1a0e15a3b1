"""Rows kept over the iterations of one reconstruction call: a call of three
iterations (rows formed in the first, read in the others) gives bit for bit
what three calls of one iteration give, for event counts around the kernel's
32-event tiles, supports that end inside a 32-voxel tile, subsets without
events, every scatter model and batches of uneven realisations."""
from __future__ import annotations

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2305_17111_gb300 as lm  # noqa: E402
from synthetic import preset, simulate  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


@pytest.mark.parametrize("name,n", [("small_24", 1), ("small_24", 31), ("small_24", 33),
                                    ("small_16", 300), ("lmmew_32", 700)])
@pytest.mark.parametrize("scatter", ["exact", "none", "surrogate_coarse"])
def test_iterations_on_kept_rows_match_recomputed_ones(name, n, scatter):
    sc = preset(name)
    ph = sc.make_phantom()
    gpu = lm.Model.from_scenario(sc, ph.rho)
    net = lm.Surrogate(3)
    gpu.set_scatter_model(scatter, net if scatter.startswith("surrogate") else None)
    lists = [simulate(sc, n_events=k, seed=70 + k) for k in (n, 2 * n + 5)]
    devs = [lm.DeviceEvents.from_list(e) for e in lists]
    lam0 = torch.from_numpy((ph.rho.reshape(-1) > 0).astype(np.float32)).cuda()
    n_sub, n_it = sc.n_subsets, 3
    want = []
    for d in devs:
        one, l1 = lam0.clone(), torch.zeros(n_it * n_sub, dtype=torch.float64, device="cuda")
        for it in range(n_it):
            gpu.osem(d, one, n_sub, it + 1, start_iter=it, loglik=l1)
        want.append((one, l1))
        all3, l3 = lam0.clone(), torch.zeros_like(l1)
        gpu.osem(d, all3, n_sub, n_it, loglik=l3)
        assert torch.equal(all3, one)
        assert torch.equal(l3, l1)
        tail = lam0.clone()      # starting inside an iteration: subsets met first later on
        gpu.osem(d, tail, n_sub, 2, 0, n_sub - 1)
        step = lam0.clone()
        gpu.osem(d, step, n_sub, 1, 0, n_sub - 1)
        gpu.osem(d, step, n_sub, 2, 1, 0)
        assert torch.equal(tail, step)
    imgs = lam0.repeat(2, 1).contiguous()
    gpu.osem_batch(devs, imgs, n_sub, n_it)
    for i in range(2):
        assert torch.equal(imgs[i], want[i][0]), f"realisation {i}"
    gpu.close()


def test_rows_beyond_a_row_block_are_given_back():
    """10 GB of kept rows (energy pruning off: the rows' route for a dense list):
    the same bits as one iteration per call, and the handle keeps no more than
    the 4 GiB a row block may take (with its eighth to spare and the sort)."""
    sc = preset("lmmew_64").with_(n_subsets=1)
    ph = sc.make_phantom()
    gpu = lm.Model.from_scenario(sc, ph.rho)
    gpu.set_energy_pruning(False)
    n = 3_000_000
    rng = np.random.default_rng(1)
    dev = lm.DeviceEvents(rng.integers(0, sc.n_angles, n), rng.integers(16, 48, n),
                          rng.uniform(60.0, 290.0, n).astype(np.float32))
    assert 4 * n * gpu.nq > 10e9
    lam0 = torch.from_numpy((ph.rho.reshape(-1) > 0).astype(np.float32)).cuda()
    both, one = lam0.clone(), lam0.clone()
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    gpu.osem(dev, both, 1, 2)
    torch.cuda.synchronize()
    assert free - torch.cuda.mem_get_info()[0] < 5.5 * 2**30
    gpu.osem(dev, one, 1, 1)
    gpu.osem(dev, one, 1, 2, 1, 0)
    assert torch.equal(both, one)
    gpu.close()


@pytest.mark.parametrize("n", [31, 300])
@pytest.mark.parametrize("form", ["surrogate", "fp16", "bf16"])
def test_other_forms_keep_the_same_rows(n, form):
    """The full surrogate and the reduced-precision forms, one call and batched."""
    sc = preset("small_24")
    ph = sc.make_phantom()
    gpu = lm.Model.from_scenario(sc, ph.rho)
    net = lm.Surrogate(3)
    if form == "surrogate":
        gpu.set_scatter_model(form, net)
    else:
        gpu.set_scatter_precision(form)
    devs = [lm.DeviceEvents.from_list(simulate(sc, n_events=k, seed=90 + k)) for k in (n, 2 * n + 5)]
    lam0 = torch.from_numpy((ph.rho.reshape(-1) > 0).astype(np.float32)).cuda()
    n_sub, n_it = sc.n_subsets, 3
    want = []
    for d in devs:
        one, l1 = lam0.clone(), torch.zeros(n_it * n_sub, dtype=torch.float64, device="cuda")
        for it in range(n_it):
            gpu.osem(d, one, n_sub, it + 1, start_iter=it, loglik=l1)
        want.append(one)
        all3, l3 = lam0.clone(), torch.zeros_like(l1)
        gpu.osem(d, all3, n_sub, n_it, loglik=l3)
        assert torch.equal(all3, one)
        assert torch.equal(l3, l1)
    imgs = lam0.repeat(2, 1).contiguous()
    gpu.osem_batch(devs, imgs, n_sub, n_it)
    for i in range(2):
        assert torch.equal(imgs[i], want[i]), f"realisation {i}"
    gpu.close()
