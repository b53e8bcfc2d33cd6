"""The resident engine's scan pieces and work split at their edges, against the oracle.

A block scans a parity's dirty bitmap in pieces of 8, 16 or 32 bits (up to 128,
256 or 512 words of 32 groups), in several rounds beyond that, and works on a
phase's groups with a lane to a point (few groups) or a thread to a group.
The heights put the bitmap of a one-block image on both sides of each line; the
widths leave one, a partial and a full last group in a row, and cross a word."""
import numpy as np
import pytest

pytest.importorskip("torch")
import torch  # noqa: E402

import oracle  # noqa: E402
from paper_1603_09180_gb300 import synth, thin  # noqa: E402

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")]


@pytest.mark.parametrize("dtype,lam", [("u8", 0), ("u8", 9), ("u16", 120)])
@pytest.mark.parametrize("h,w", [(256, 24), (258, 25), (512, 17), (514, 23), (1024, 9), (1026, 10), (64, 258), (96, 520)])
def test_scan_pieces(h, w, dtype, lam):
    n = torch.cuda.get_device_properties(0).multi_processor_count + 1  # so many images that none is spread over blocks
    img = synth.value_noise_image(h, w, dtype, seed=3 * h + w)
    ref, _ = oracle.thin(img, lam)
    imgs = [torch.from_numpy(img).cuda() for _ in range(n)]
    stats, _ = thin.batch(imgs, [lam] * n)
    torch.cuda.synchronize()
    assert all(s["converged"] == 1 for s in stats)
    for t in imgs[:: n - 1]:
        assert np.array_equal(t.cpu().numpy(), ref)
