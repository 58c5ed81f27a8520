"""The FP64 march computes only the part of each window that lies in the domain and that the source has reached: kernels
of every source against the oracle where those limits bite -- windows larger than the domain on one, two and all axes,
substep counts around the radius, and batches that mix fully and partly covered windows."""
import numpy as np
import pytest

import oracle
from paper_2408_11376_gb300 import FDiRW, synth

pytestmark = pytest.mark.gpu
KERNEL_TOL = 1e-13               # per-kernel relative L2, as the other FP64 kernel tests


@pytest.fixture(scope="module", autouse=True)
def _library():
    from paper_2408_11376_gb300 import build
    build.build()


@pytest.mark.parametrize("shape,R,n_sub", [((5, 4, 3), 8, 1), ((5, 4, 3), 8, 30), ((1, 1, 12), 5, 7), ((12, 2, 1), 3, 2),
                                           ((3, 14, 6), 4, 4), ((9, 8, 7), 1, 3), ((11, 10, 9), 2, 6), ((17, 9, 6), 6, 25),
                                           ((13, 12, 11), 7, 3)])
def test_every_kernel_matches_the_oracle(shape, R, n_sub):
    D = synth.random_diffusivity(shape, 200 + R, 4.0)
    lam = oracle.stable_dt_sub(shape, D)
    N = int(np.prod(shape))
    src = np.arange(N)
    with FDiRW(shape, D, n_sub * lam, R, n_sub, "fp64") as f:
        f.kernels()
        ks = f.read_kernels(src).reshape(N, -1)
    ref, _ = oracle.kernels(shape, D, lam, R, n_sub, src)
    ref = ref.reshape(N, -1)
    err = np.linalg.norm(ks - ref, axis=1) / np.linalg.norm(ref, axis=1)
    assert err.max() <= KERNEL_TOL
    assert np.max(np.abs(ks.sum(axis=1) - 1.0)) <= 1e-12
