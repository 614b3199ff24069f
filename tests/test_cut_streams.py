"""Carried rows: the kernels take each row of a frame from the carried or from the new samples (a
tensor-core build task 8 times of a block, a producer warp of the FP32 form 4 rows).  A stream cut at
any sample (inside such a group, at a block's edge, one short of a frame, several cuts) gives the bits
of the uncut one."""
import numpy as np
import pytest

from paper_1702_04728_gb300 import binding as B
from paper_1702_04728_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cuts", [(1,), (5,), (64,), (127,), (128,), (261,), (383,), (384 + 130,), (3, 390, 1000)])
@pytest.mark.parametrize("form", [B.BF_FP32_FFT, B.BF_TC_DFT256, B.BF_TC_DFT256_X2, B.BF_TC_DFT256_X1])
def test_cut_streams_have_the_bits_of_the_whole(built_lib, form, cuts):
    freqs = [430e6, 760e6]
    n = 384 * 4 + 77
    rng = np.random.default_rng(29)
    raw = synth.encode(rng.integers(-7, 8, size=(2, n, 2048)), rng.integers(-7, 8, size=(2, n, 2048)))
    raw = torch.from_numpy(raw).cuda()
    edges = [0, *cuts, n]
    with B.Plan(form=form) as p:
        whole = p.run(raw, freqs, stream_id=1)
        got = [p.run(raw[:, a:b].contiguous(), freqs, stream_id=2, flags=B.BF_END_OF_STREAM if b == n else 0)
               for a, b in zip(edges, edges[1:])]
    assert torch.equal(torch.cat(got, dim=2), whole)
