"""The mosaic engine (a few images, a block to a tile, rims exchanged through flags) against the oracle.

Sizes with one tile, tiles that end at, inside and one pixel past the image, rows that do not start at
16-byte boundaries; caps and resumes inside a step; 16 images (the most that take it) and 17."""
import numpy as np
import pytest

pytest.importorskip("torch")
import torch  # noqa: E402

import oracle  # noqa: E402
from paper_1603_09180_gb300 import synth, thin  # noqa: E402

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")]


@pytest.mark.parametrize("h,w,dtype,lam,op,adj", [
    (3, 3, "u8", 4, "thinning", 0), (16, 32, "u8", 0, "thinning", 0), (17, 33, "u16", 60, "thinning", 0),
    (128, 256, "u8", 12, "thinning", 0), (129, 257, "u8", 12, "skeleton", 0), (33, 700, "u16", 200, "thinning", 1),
    (600, 35, "u8", 0, "skeleton", 1), (3, 30000, "u8", 8, "thinning", 0), (511, 513, "u8", 3, "thinning", 0)])
def test_mosaic(h, w, dtype, lam, op, adj):
    img = synth.value_noise_image(h, w, dtype, seed=2 * h + w)
    ref, rst = oracle.thin(img, lam, op={"thinning": 0, "skeleton": 1}[op], adj=adj)
    base = torch.from_numpy(img).cuda()
    for pad, at in ((0, 0), (5, 3)):  # packed rows, then rows at odd addresses
        t = torch.empty((h, w + pad), dtype=base.dtype, device="cuda")[:, at:at + w]
        t.copy_(base)
        st = thin.run(t, lam, op=op, adj=adj)
        assert np.array_equal(t.cpu().numpy(), ref)
        assert st["converged"] == 1 and st["lowered"] == rst["lowered"] and st["last_change_phase"] == rst["last_change_phase"]
    t = base.clone()
    g, low = 0, 0
    for cap in (1, 2, 14, 15, 16, -1):
        st = thin.run(t, lam, op=op, adj=adj, start_phase=g, max_phases=cap)
        assert cap < 0 or st["phases"] <= cap
        g, low = st["end_phase"], low + st["lowered"]
    assert np.array_equal(t.cpu().numpy(), ref) and low == rst["lowered"]


@pytest.mark.parametrize("n", [2, 16, 17])
def test_few_images(n):
    shapes = [(40 + 17 * k, 90 + 11 * k) for k in range(n)]
    imgs = [synth.value_noise_image(h, w, "u8", seed=h) for h, w in shapes]
    lams = [(0, 6, 15)[k % 3] for k in range(n)]
    work = [torch.from_numpy(a).cuda() for a in imgs]
    stats, rc = thin.batch(work, lams)
    assert rc == 0
    for a, lam, t, st in zip(imgs, lams, work, stats):
        ref, rst = oracle.thin(a, lam)
        assert np.array_equal(t.cpu().numpy(), ref)
        assert st["lowered"] == rst["lowered"] and st["last_change_phase"] == rst["last_change_phase"]


def test_set_tile_shape_is_still_checked():
    """Images that fit the mosaic's tiles but no cluster, with a depth that no u16 call takes: refused, untouched."""
    img = synth.value_noise_image(1500, 1500, "u16", seed=1)
    work = [torch.from_numpy(img).cuda() for _ in range(3)]
    with pytest.raises(thin.ThinError):
        thin.batch(work, [60] * 3, halo=9)
    assert all(np.array_equal(t.cpu().numpy(), img) for t in work)


def _naive(img, lam):
    """The phases one launch after another, straight from global memory (no tiles)."""
    t = torch.from_numpy(img).cuda()
    st = thin.run(t, lam, kernel="naive")
    return t, st


@pytest.mark.parametrize("h,w,lams,n", [(1548, 1470, (0, 80), 1), (965, 693, (0, 80), 1), (794, 870, (40,), 1), (2000, 2000, (0,), 1),
                                        (2048, 2048, (0, 30), 1), (1200, 1200, (30,), 4), (700, 700, (30,), 16)])
def test_high_u16_tiles(h, w, lams, n):
    """u16 images whose tiles are 200 to 300 rows high, several side by side."""
    for lam in lams:
        imgs = [synth.value_noise_image(h, w, "u16", seed=h + w + k) for k in range(min(n, 2))]
        want = [_naive(im, lam) for im in imgs]
        work = [torch.from_numpy(imgs[k % len(imgs)]).cuda() for k in range(n)]
        stats, rc = thin.batch(work, [lam] * n)
        assert rc == 0
        for k, (t, st) in enumerate(zip(work, stats)):
            ref, rst = want[k % len(imgs)]
            assert st["tiles_visited"] == 0 and st["converged"] == 1
            assert torch.equal(t.view(torch.int16), ref.view(torch.int16))
            assert st["lowered"] == rst["lowered"] and st["last_change_phase"] == rst["last_change_phase"]


def test_high_u16_tiles_against_the_oracle():
    img = synth.value_noise_image(965, 693, "u16", seed=9)
    ref, rst = oracle.thin(img, 0)
    t = torch.from_numpy(img).cuda()
    st = thin.run(t, 0)
    assert np.array_equal(t.cpu().numpy(), ref)
    assert st["lowered"] == rst["lowered"] and st["last_change_phase"] == rst["last_change_phase"]
