"""The tiled engine's tiles at their edges, against the oracle: the smallest tile, tiles of one and of two
TMA boxes, the longest steps, images that end inside, at and just past a tile, caps and resumes inside a step."""
import numpy as np
import pytest

pytest.importorskip("torch")
import torch  # noqa: E402

import oracle  # noqa: E402
from paper_1603_09180_gb300 import synth, thin  # noqa: E402

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")]


@pytest.mark.parametrize("tile,halo", [(None, 0), ((16, 8), 3), ((32, 18), 16), ((224, 240), 8), ((208, 240), 7)])
@pytest.mark.parametrize("h,w,dtype,lam", [(241, 225, "u8", 7), (240, 224, "u8", 0), (97, 241, "u16", 90), (9, 17, "u8", 5)])
def test_tiles(h, w, dtype, lam, tile, halo):
    if dtype == "u16" and halo > 8:
        pytest.skip("u16 takes steps of at most 8 phases")
    img = synth.value_noise_image(h, w, dtype, seed=h + 5 * w)
    ref, rst = oracle.thin(img, lam)
    t = torch.from_numpy(img).cuda()
    st = thin.run(t, lam, kernel="tiled", tile=tile, halo=halo)
    assert np.array_equal(t.cpu().numpy(), ref)
    assert st["converged"] == 1 and st["lowered"] == rst["lowered"] and st["last_change_phase"] == rst["last_change_phase"]
    t = torch.from_numpy(img).cuda()
    at = 0
    for cap in (1, 2, 9, -1):
        at = thin.run(t, lam, kernel="tiled", tile=tile, halo=halo, start_phase=at, max_phases=cap)["end_phase"]
    assert np.array_equal(t.cpu().numpy(), ref)


@pytest.mark.parametrize("op,adj", [("thinning", 0), ("skeleton", 1)])
@pytest.mark.parametrize("h,w,dtype,tile,halo", [
    (759, 1009, "u8", (32, 32), 8), (1601, 805, "u16", (64, 32), 4), (789, 785, "u8", (16, 8), 3), (785, 789, "u16", (16, 8), 3),
    (1800, 1501, "u8", (32, 16), 15), (1220, 515, "u8", (32, 32), 16)])
def test_many_small_tiles(h, w, dtype, tile, halo, op, adj):
    """So many tiles that blocks of 4 or of 2 warps take them."""
    img = synth.value_noise_image(h, w, dtype, seed=h)
    lam = 0 if dtype == "u8" else 40
    ref, rst = oracle.thin(img, lam, op={"thinning": 0, "skeleton": 1}[op], adj=adj)
    t = torch.from_numpy(img).cuda()
    st = thin.run(t, lam, kernel="tiled", tile=tile, halo=halo, op=op, adj=adj)
    assert np.array_equal(t.cpu().numpy(), ref)
    assert st["converged"] == 1 and st["lowered"] == rst["lowered"] and st["last_change_phase"] == rst["last_change_phase"]


@pytest.mark.parametrize("n", [23, 24])
def test_many_cluster16_images_go_to_tiles(n):
    """24 images that need a cluster of 16 blocks go to the tiled engine, 23 do not; the result is the same."""
    imgs = [synth.value_noise_image(1300, 1310, "u8", seed=s) for s in (1, 2)]
    want = []
    for im in imgs:
        t = torch.from_numpy(im).cuda()
        thin.run(t, 3, kernel="resident")
        want.append(t)
    work = [torch.from_numpy(imgs[k % 2]).cuda() for k in range(n)]
    stats, rc = thin.batch(work, [3] * n)
    assert rc == 0
    assert all((s["tiles_visited"] > 0) == (n >= 24) for s in stats)
    for k, t in enumerate(work):
        assert torch.equal(t, want[k % 2])


@pytest.mark.parametrize("n", [17, 40, 60])
@pytest.mark.parametrize("h,w,dtype", [(1030, 311, "u8"), (632, 351, "u16"), (256, 1366, "u8"), (300, 300, "u8")])
def test_spread_clusters(h, w, dtype, n):
    """Images that need clusters of 3 (and smaller ones), so few that each is spread over a wider cluster."""
    img = synth.value_noise_image(h, w, dtype, seed=h + w)
    want = torch.from_numpy(img).cuda()
    thin.run(want, 4, kernel="tiled")
    work = [torch.from_numpy(img).cuda() for _ in range(n)]
    stats, rc = thin.batch(work, [4] * n)
    assert rc == 0 and all(s["tested"] > 0 and s["converged"] == 1 for s in stats)
    for t in work:
        assert torch.equal(t.view(torch.uint8), want.view(torch.uint8))
