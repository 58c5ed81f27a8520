"""The 2x2-block march (mapping 4) against a one-column-per-thread mapping, bit for bit, where its level pairs,
partial batches, window clipping and both z parts can go wrong: every radius, odd and even substep counts down to
none, source counts that fill the last batch and do not, every storage type, and the z-slabs of a streamed cache."""
import numpy as np
import pytest
import torch

from paper_2408_11376_gb300 import FDiRW, fdirw, synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module", autouse=True)
def _library():
    from paper_2408_11376_gb300 import build
    build.build()


def _run(shape, D, dt, R, n_sub, prec, parts, mem_limit=0):
    N = int(np.prod(shape))
    c0 = torch.from_numpy(synth.random_field(N, 5)).to(DEV)
    out = torch.empty_like(c0)
    with FDiRW(shape, D, n_sub * dt, R, n_sub, prec, march_parts=parts, mem_limit=mem_limit) as f:
        f.step(c0, out, 2)
        info = f.info()
        ks = None if info["n_chunks"] > 1 else f.read_kernels(np.arange(N))
    return out.cpu().numpy(), ks, info


@pytest.mark.parametrize("R", range(1, 11))
@pytest.mark.parametrize("n_sub,prec,shape", [(0, "fp32", (5, 4, 3)), (1, "fp32", (13, 5, 7)), (2, "bf16", (7, 11, 9)),
                                              (9, "fp16", (12, 10, 23))])
def test_block_march_equals_the_column_march(R, n_sub, prec, shape):
    D = synth.random_diffusivity(shape, 7 + R, 6.0)
    dt = fdirw.fdirw_stable_dt(shape, D)
    other = 1 if R <= 8 else 5
    a, ka, ia = _run(shape, D, dt, R, n_sub, prec, 4)
    b, kb, ib = _run(shape, D, dt, R, n_sub, prec, other)
    assert (ia["march_parts"], ib["march_parts"]) == (4, other)
    assert np.array_equal(ka, kb) and np.array_equal(a, b)
    assert np.max(np.abs(ka.reshape(len(ka), -1).sum(axis=1) - 1.0)) <= 1e-12


@pytest.mark.parametrize("R", [3, 8, 10])
def test_block_march_streams_slabs(R):
    shape = (10, 9, 26)
    D = synth.random_diffusivity(shape, 70 + R, 4.0)
    dt = fdirw.fdirw_stable_dt(shape, D)
    a, _, ia = _run(shape, D, dt, R, 6, "bf16", 4)
    limit = ia["device_bytes"] - ia["cache_bytes"] + ia["cache_bytes"] // 4 + 8 * int(np.prod(shape))
    b, _, ib = _run(shape, D, dt, R, 6, "bf16", 4, mem_limit=limit)
    assert ib["n_chunks"] > 1 and np.array_equal(a, b)
