"""Work units of a launch: a request whose last (or only) round of items would leave CTAs idle runs
them in parts of 1, 2 or 3 of an item's six passes.  Every output adds the six passes in one fixed
order, so each frame must have the same bits whatever the length of its request.  The frame counts
give, on 152 SMs (152 CTAs, 76 CTA pairs): parts of every size, with and without whole items beside
them, and no parts."""
import numpy as np
import pytest

from paper_1702_04728_gb300 import binding as B
from paper_1702_04728_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form", [B.BF_FP32_FFT, B.BF_TC_DFT256, B.BF_TC_DFT256_X2, B.BF_TC_DFT256_X1,
                                  B.BF_TC_DFT512])
def test_frames_do_not_depend_on_the_request_length(built_lib, form):
    freqs = [455e6, 705e6]
    rng = np.random.default_rng(17)
    raw = synth.encode(rng.integers(-7, 8, size=(2, 384 * 41, 2048)), rng.integers(-7, 8, size=(2, 384 * 41, 2048)))
    raw = torch.from_numpy(raw).cuda()
    with B.Plan(form=form) as p:
        whole = p.run(raw, freqs)
        for n_chan, nf in ((1, 1), (1, 2), (1, 8), (1, 13), (1, 19), (1, 25), (1, 37), (1, 39), (2, 1), (2, 20)):
            out = p.run(raw[:n_chan, : 384 * nf].contiguous(), freqs[:n_chan])
            assert torch.equal(out, whole[:, : 16 * n_chan, :nf]), f"{n_chan} channels x {nf} frames"
