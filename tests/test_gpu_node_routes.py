"""Which route a call takes (csrc/api.cu) follows the model, the forms set on the
handle and the list's length alone.  The scatter grid of 80 x 80 cells has node
sums of one angle that the no-allocation call's array does not hold, where
lm_forward has to keep the rows that lm_forward_noalloc may run; the tile size,
which the autotuner and lm_set_tile_events change, has no say in any route, and
the array none in back projections and reconstructions."""
from __future__ import annotations

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2305_17111_gb300 as lm  # noqa: E402
from synthetic import preset  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


def _events(sc, n, seed):
    rng = np.random.default_rng(seed)
    return lm.DeviceEvents(rng.integers(0, sc.n_angles, n), rng.integers(16, 48, n),
                           rng.uniform(70.0, 280.0, n).astype(np.float32))


@pytest.fixture(scope="module")
def big():
    sc = preset("lmmew_64").with_(n=80, pixel_cm=0.4, scatter_n=80)
    rho = sc.make_phantom().rho
    gpu = lm.Model.from_scenario(sc, rho)
    lam = torch.from_numpy((rho.reshape(-1) > 0).astype(np.float32)).cuda()
    yield sc, gpu, lam
    gpu.close()


def _on_nodes(gpu, call, launches):
    """The result and whether `launches` path kernels of the node route ran."""
    gpu.profile_enable(True)
    out = call()
    terms = gpu.profile_read()["terms"]
    gpu.profile_enable(False)
    return out, terms == launches * gpu.n_lines * gpu.nq * gpu.np_scatter


def test_tile_size_has_no_say(big):
    sc, gpu, lam = big
    dev = _events(sc, 40_000, 1)
    w = torch.rand(40_000, device="cuda", generator=torch.Generator("cuda").manual_seed(1))

    def osem():
        img = lam.clone()
        gpu.osem(dev, img, 10, 1)
        return img

    got = {}
    for tile in (128, 32):
        gpu.set_tile_events(tile)
        img, nodes = _on_nodes(gpu, osem, 20)            # forward and back, 10 subsets
        assert nodes
        bp, nodes = _on_nodes(gpu, lambda: gpu.backproject(dev, w), 1)
        assert nodes
        y, nodes = _on_nodes(gpu, lambda: gpu.forward(dev, lam), 1)
        assert not nodes                                 # 40 000 rows fit the array in 32-event tiles
        got[tile] = (img, bp, y)
    out = torch.empty_like(got[32][2])
    gpu.forward_noalloc(dev, lam, out)
    assert torch.equal(out, got[32][2])
    for a, b in zip(got[128], got[32]):
        assert torch.equal(a, b)
    y, nodes = _on_nodes(gpu, lambda: gpu.forward(_events(sc, 120_000, 2), lam), 1)
    assert nodes                                         # more than the array holds in any tile
    with pytest.raises(lm.LmmewError, match="INVALID_ARG"):
        gpu.forward_noalloc(_events(sc, 120_000, 2), lam, torch.empty(120_000, device="cuda"))


def test_batch_reconstructs_every_realisation_after_a_retune(big):
    sc, gpu, lam = big
    lists = [_events(sc, n, 10 + n) for n in (40_000, 3_000, 60_000)]
    gpu.set_tile_events(128)
    want = []
    for d in lists:
        img = lam.clone()
        gpu.osem(d, img, 10, 1)
        want.append(img)
    for tile in (128, 32):
        gpu.set_tile_events(tile)
        imgs = lam.repeat(3, 1).contiguous()
        gpu.osem_batch(lists, imgs, 10, 1)
        for i in range(3):
            assert torch.equal(imgs[i], want[i]), f"realisation {i}, {tile}-event tiles"


def test_noalloc_goes_through_blocks_of_angles():
    """The 64 x 64 scanner: a few angles' node sums at a time in the array."""
    sc = preset("lmmew_64")
    rho = sc.make_phantom().rho
    gpu = lm.Model.from_scenario(sc, rho)
    dev = _events(sc, 4_000, 5)
    lam = torch.from_numpy((rho.reshape(-1) > 0).astype(np.float32)).cuda()
    y, nodes = _on_nodes(gpu, lambda: gpu.forward(dev, lam), 1)
    assert nodes
    out = torch.empty_like(y)
    gpu.forward_noalloc(dev, lam, out)
    assert torch.equal(out, y)
    gpu.close()


def test_a_reconstruction_keeps_its_route_when_memory_is_short():
    """80 MiB free, where the node sums of all 24 angles at once take 120: the
    same bits as with all of the memory (in smaller blocks), not the rows."""
    sc = preset("lmmew_64").with_(n_angles=24, n_subsets=1)
    rho = sc.make_phantom().rho
    dev = _events(sc, 6_000, 3)
    lam = torch.from_numpy((rho.reshape(-1) > 0).astype(np.float32)).cuda()
    want, got = lam.clone(), lam.clone()
    gpu = lm.Model.from_scenario(sc, rho)
    gpu.osem(dev, want, 1, 2)
    gpu.close()
    gpu = lm.Model.from_scenario(sc, rho)
    gpu.set_tile_events(32)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    rest = torch.empty(torch.cuda.mem_get_info()[0] - (80 << 20), dtype=torch.uint8, device="cuda")
    try:
        gpu.osem(dev, got, 1, 2)
    finally:
        del rest
        torch.cuda.empty_cache()
    assert torch.equal(got, want)
    gpu.close()
