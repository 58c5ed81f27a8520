"""Gathers of one field that run different kernels, because a streamed cache has fewer destinations a launch than the
resident one or packed rows in the place of padded ones: the same bits."""
import numpy as np
import pytest
import torch

from paper_2408_11376_gb300 import FDiRW, fdirw, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _library():
    from paper_2408_11376_gb300 import build
    build.build()


@pytest.mark.parametrize("shape,R,prec,accum", [((48, 40, 40), 1, "bf16", "ff"), ((48, 40, 40), 1, "fp16", "fp32"),
                                                ((88, 80, 76), 3, "bf16", "fp32"), ((83, 80, 81), 3, "fp16", "fp32"),
                                                ((83, 20, 19), 4, "fp32", "ff"), ((21, 20, 19), 6, "bf16", "ff")])
def test_streamed_gather_equals_the_resident_one(shape, R, prec, accum):
    N = int(np.prod(shape))
    D = synth.random_diffusivity(shape, 50 + R, 3.0)
    dt = fdirw.fdirw_stable_dt(shape, D)
    c = torch.from_numpy(synth.random_field(N, 51, -1.0, 1.0)).cuda()
    out, info, limit = [], [], 0
    for _ in range(2):
        with FDiRW(shape, D, 4 * dt, R, 4, prec, accum=accum, mem_limit=limit) as f:
            out.append(torch.empty_like(c))
            f.step(c, out[-1], 2)
            info.append(f.info())
        i = info[0]
        limit = i["device_bytes"] - i["cache_bytes"] + i["cache_bytes"] // 3 + 8 * N
    assert info[0]["n_chunks"] == 1 and info[1]["n_chunks"] >= 3
    assert torch.equal(out[0], out[1])
