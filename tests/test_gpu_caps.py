"""The status of a default call at a phase cap.  Whichever engine takes the images, the call converged if
the last three phases changed nothing (the rule of the resident engine), also where the engine's own
bookkeeping already knows, or does not know yet, that no point is left to test."""
import numpy as np
import pytest

pytest.importorskip("torch")
import torch  # noqa: E402

from paper_1603_09180_gb300 import synth, thin  # noqa: E402

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")]

FIELDS = ("rc", "status", "converged", "lowered", "last_change_phase")


def _peak():
    a = np.zeros((3, 3), np.uint8)
    a[1, 1], a[0, 1] = 5, 9  # the only interior point: lowered in phase 3, no neighbour to test again
    return a


@pytest.mark.parametrize("img,lam", [(_peak(), 0), (synth.value_noise_image(64, 64, "u8", seed=0), 10),
                                     (synth.value_noise_image(200, 200, "u8", seed=1), 0)])
@pytest.mark.parametrize("start", [0, 5])
def test_one_image(img, lam, start):
    full = thin.run(torch.from_numpy(img).cuda(), lam, start_phase=start)
    last = full["last_change_phase"] - start
    for cap in list(range(1, 12)) + list(range(max(last - 3, 12), last + 22)):
        got, want = (thin.run(torch.from_numpy(img).cuda(), lam, start_phase=start, max_phases=cap, check=False, kernel=k)
                     for k in ("auto", "resident"))
        assert [got[f] for f in FIELDS] == [want[f] for f in FIELDS], cap
        assert got["converged"] == int(cap >= 4 and got["last_change_phase"] < start + cap - 3)
        assert got["phases"] <= cap and got["end_phase"] == start + got["phases"]
        if not got["converged"]:
            assert got["end_phase"] == start + cap


@pytest.mark.parametrize("cap", [1 << 40, (1 << 63) - 1])
def test_caps_out_of_reach(cap):
    img = synth.value_noise_image(64, 64, "u8", seed=0)
    full = thin.run(torch.from_numpy(img).cuda(), 10, start_phase=5)
    for kernel in ("auto", "resident"):
        st = thin.run(torch.from_numpy(img).cuda(), 10, start_phase=5, max_phases=cap, check=False, kernel=kernel)
        assert [st[f] for f in FIELDS] == [full[f] for f in FIELDS]


def test_batch_that_goes_to_tiles():
    img = torch.from_numpy(synth.value_noise_image(1300, 1310, "u8", seed=1)).cuda()
    last = thin.run(img.clone(), 0, kernel="resident")["last_change_phase"]
    for cap in (3, 15, last + 1, last + 2, last + 3, last + 4, last + 5, last + 9, last + 19):
        want = thin.run(img.clone(), 0, kernel="resident", max_phases=cap, check=False)
        stats, rc = thin.batch([img.clone() for _ in range(24)], [0] * 24, max_phases=cap, check=False)
        assert rc == want["rc"] and all(s["tiles_visited"] > 0 for s in stats)
        for s in stats:
            assert [s[f] for f in FIELDS[1:]] == [want[f] for f in FIELDS[1:]], cap
            assert s["phases"] <= cap and (s["converged"] or s["end_phase"] == cap)
