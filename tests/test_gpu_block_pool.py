"""Device blocks that a destroyed context leaves to the next one: results do not depend on what a block held before,
contexts of several threads on their own streams share the pool, and what it keeps is bounded."""
import threading

import numpy as np
import pytest
import torch

from paper_2408_11376_gb300 import FDiRW, FDiRWCoarse, fdirw, synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module", autouse=True)
def _library():
    from paper_2408_11376_gb300 import build
    build.build()


def _job(shape, seed, prec, accum, stream=None):
    D = synth.random_diffusivity(shape, seed, 3.0)
    dt = fdirw.fdirw_stable_dt(shape, D)
    out = np.empty(D.size)
    with FDiRW(shape, D, 8 * dt, 3, 8, prec, accum=accum, stream=stream) as f:
        assert f.info()["last_restore_drift"] == 0.0
        f.step(synth.random_field(D.size, seed), out, 2)
    return out


CASES = [((12, 11, 10), 1, "fp32", "ff"), ((12, 11, 10), 2, "bf16", "fp32"), ((9, 14, 8), 3, "fp64", "ff"),
         ((17, 6, 13), 4, "fp16", "fp32"), ((12, 11, 10), 1, "fp32", "ff")]


def test_reused_blocks_change_nothing():
    first = [_job(*c) for c in CASES]
    for _ in range(3):
        for c, want in zip(CASES, first):
            assert np.array_equal(_job(*c), want)
        with FDiRWCoarse((12, 11, 10), np.ones(1320), None, 3, 0.5, 3, 4) as f:    # leaves blocks of other contents
            f.far_field(50.0, 0.1)
            f.step(np.ones(1320), np.empty(1320), 1)


def test_contexts_of_several_threads_share_the_pool():
    want = [_job(*c) for c in CASES]
    bad = []

    def work(k):
        s = torch.cuda.Stream(device=DEV)
        for i in range(6):
            c = (k + i) % len(CASES)
            if not np.array_equal(_job(*CASES[c], stream=s), want[c]):
                bad.append((k, i))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad


def test_what_stays_is_bounded():
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info(0)[0]
    for n in (40, 48, 56, 64, 60, 52, 44):
        shape = (n,) * 3
        D = np.ones(n ** 3)
        with FDiRW(shape, D, 0.5, 4, 4, "bf16") as f:
            f.kernels()
    torch.cuda.synchronize()
    assert free0 - torch.cuda.mem_get_info(0)[0] <= (256 << 20) + (64 << 20)     # 256 MB and the driver's own granularity
