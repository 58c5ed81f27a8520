"""The coarse step's mapping and gather at block counts on either side of where their kernels change, with one cell a
block and with few and many offsets, against the same sums in numpy on the matrix that the library stored."""
import numpy as np
import pytest

from paper_2408_11376_gb300 import FDiRWCoarse, fdirw, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _library():
    from paper_2408_11376_gb300 import build
    build.build()


@pytest.mark.parametrize("B,R,shape", [(1, 1, (33, 37, 10)), (1, 1, (35, 34, 34)), (1, 3, (36, 34, 33)), (3, 2, (66, 67, 71)),
                                       (3, 2, (67, 68, 72)), (3, 5, (104, 103, 100)), (5, 3, (19, 16, 13)), (7, 0, (30, 29, 8))])
def test_coarse_step_sums(B, R, shape):
    nx, ny, nz = shape
    rng = np.random.default_rng(B + R)
    liquid = (rng.random(nx * ny * nz) < 0.6).astype(np.uint8)
    D = np.where(liquid, rng.uniform(0.3, 1.0, liquid.size), 1e-6)
    dt = fdirw.fdirw_stable_dt(shape, D)
    nc = [-(-n // B) for n in shape]
    c = synth.random_field(D.size, 8, -1.0, 2.0)
    out = np.empty_like(c)
    with FDiRWCoarse(shape, D, liquid, B, 3 * dt, R, 3) as f:
        f.step(c, out)
        P = f.read_coarse(np.arange(np.prod(nc)))                 # [J, d]: to block J + d
    z, y, x = np.meshgrid(*(np.arange(n) for n in (nz, ny, nx)), indexing="ij")
    block = (((z // B) * nc[1] + y // B) * nc[0] + x // B).reshape(-1)
    lq = liquid.astype(bool)
    count = np.bincount(block[lq], minlength=np.prod(nc))
    mean = np.bincount(block[lq], c[lq], np.prod(nc)) / np.maximum(count, 1)
    size = np.bincount(block[lq], np.abs(c[lq]), np.prod(nc)) / np.maximum(count, 1)

    def spread(P, C):
        Rc = P.shape[1] // 2
        cx, cy, cz = nc
        to = np.zeros((cz + 2 * Rc, cy + 2 * Rc, cx + 2 * Rc))
        for k in range(2 * Rc + 1):
            for j in range(2 * Rc + 1):
                for i in range(2 * Rc + 1):
                    to[k:k + cz, j:j + cy, i:i + cx] += (P[:, k, j, i] * C).reshape(cz, cy, cx)
        return to[Rc:Rc + cz, Rc:Rc + cy, Rc:Rc + cx].reshape(-1)
    want = np.where(lq, spread(P, mean)[block], c)
    # at most B^3 + (2 Rc + 1)^3 roundings of terms that add up to `bound`
    bound = np.where(lq, spread(np.abs(P), size)[block], np.abs(c))
    assert np.all(np.abs(out - want) <= (B ** 3 + P[0].size) * 2.0 ** -52 * bound)
