"""Radii 9 and 10 with enough sources that they are stored in groups (four of 16-bit values, two of 32): groups that the
last sources do not fill, every storage type, and groups in the slabs of a streamed cache, against the one-column march
and the resident cache bit for bit."""
import numpy as np
import pytest
import torch

from paper_2408_11376_gb300 import FDiRW, fdirw, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _library():
    from paper_2408_11376_gb300 import build
    build.build()


def _run(shape, D, dt, R, prec, parts, limit=0):
    c = torch.from_numpy(synth.random_field(D.size, 9)).cuda()
    out = torch.empty_like(c)
    src = np.concatenate([np.arange(0, D.size, 37), np.arange(D.size - 9, D.size)])
    with FDiRW(shape, D, 4 * dt, R, 4, prec, march_parts=parts, mem_limit=limit) as f:
        f.step(c, out, 1)
        i = f.info()
        return out, f.read_kernels(src) if i["n_chunks"] == 1 else None, i


@pytest.mark.parametrize("R", [9, 10])
@pytest.mark.parametrize("shape,prec", [((19, 18, 19), "fp16"), ((23, 13, 21), "bf16"), ((15, 15, 15), "fp32"),
                                        ((20, 20, 17), "bf16")])
def test_grouped_stores_equal_the_column_march(R, shape, prec):
    D = synth.random_diffusivity(shape, 40 + R, 4.0)
    dt = fdirw.fdirw_stable_dt(shape, D)
    a, ka, _ = _run(shape, D, dt, R, prec, 4)
    b, kb, _ = _run(shape, D, dt, R, prec, 5)
    assert torch.equal(a, b) and np.array_equal(ka, kb)


@pytest.mark.parametrize("prec", ["fp32", "bf16"])
def test_grouped_stores_stream_slabs(prec):
    shape, R = (17, 19, 40), 9
    D = synth.random_diffusivity(shape, 44, 4.0)
    dt = fdirw.fdirw_stable_dt(shape, D)
    a, _, i = _run(shape, D, dt, R, prec, 4)
    limit = i["device_bytes"] - i["cache_bytes"] + i["cache_bytes"] // 2 + 8 * D.size
    b, _, j = _run(shape, D, dt, R, prec, 4, limit)
    assert i["n_chunks"] == 1 and j["n_chunks"] > 1 and torch.equal(a, b)
