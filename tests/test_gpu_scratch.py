"""Default calls where scratch runs out (THIN_SCRATCH_MAX bounds an allocation): images that fit a cluster
or the wide mode are thinned there, with next to no scratch; a call that fits nowhere is refused with its
images untouched."""
import numpy as np
import pytest

pytest.importorskip("torch")
import torch  # noqa: E402

from paper_1603_09180_gb300 import synth, thin  # noqa: E402

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")]


@pytest.mark.parametrize("h,w,dtype,n,most", [(200, 210, "u8", 1, 20 << 10), (300, 310, "u16", 16, 1 << 20),
                                              (1700, 1700, "u8", 1, 3 << 20), (1300, 1310, "u8", 24, 8 << 20)])
@pytest.mark.parametrize("runner", ["batch", "plan"])
def test_spares_scratch(monkeypatch, runner, h, w, dtype, n, most):
    img = torch.from_numpy(synth.value_noise_image(h, w, dtype, seed=h)).cuda()
    want = img.clone()
    wst = thin.run(want, 3, kernel="naive")
    monkeypatch.setenv("THIN_SCRATCH_MAX", str(most))
    work = [img.clone() for _ in range(n)]
    if runner == "batch":
        stats, rc = thin.batch(work, [3] * n)
    else:
        plan = thin.GraphPlan(work, [3] * n)
        stats, rc = plan.run(stats=True)
        assert plan.tiling() == (0, 0, 0)
        plan.close()
    assert rc == 0
    for t, st in zip(work, stats):
        assert torch.equal(t.view(torch.uint8), want.view(torch.uint8))
        assert st["tiles_visited"] == 0 and st["lowered"] == wst["lowered"]
        assert st["last_change_phase"] == wst["last_change_phase"] and st["converged"] == 1


@pytest.mark.parametrize("h,w,n", [(200, 210, 1), (1300, 1310, 24)])
def test_refused_untouched(monkeypatch, h, w, n):
    img = torch.from_numpy(synth.value_noise_image(h, w, "u8", seed=h)).cuda()
    work = [img.clone() for _ in range(n)]
    monkeypatch.setenv("THIN_SCRATCH_MAX", "100")
    with pytest.raises(thin.ThinError) as e:
        thin.batch(work, [3] * n)
    assert e.value.code == thin.THIN_ERR_OOM
    monkeypatch.delenv("THIN_SCRATCH_MAX")
    assert all(torch.equal(t, img) for t in work)
    thin.batch(work, [3] * n)  # and the next call works
