"""The training loss when its terms are summed in parts on two streams: against its formula evaluated from the traced head
values, for batches from one source to more than one wave of blocks, with zero targets, and from call to call."""
import numpy as np
import pytest

from oracle import surrogate as so
from paper_2408_11376_gb300 import FDiRW, Net, fdirw, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _library():
    from paper_2408_11376_gb300 import build
    build.build()


@pytest.mark.parametrize("n", [1, 2, 153, 301])
def test_loss_of_parts(n):
    # Each of the <= 301 x 4913 terms is a few FP64 roundings off (exp, log, three products and sums: <= 8 x 2^-53 of
    # its parts), sums over parts grow that by less than the 2^21 terms' pairwise depth of 32: below 1e-12 of the sum of parts.
    shape = (21, 19, 17)
    N = int(np.prod(shape))
    src = np.random.default_rng(n).choice(N, n, replace=False).astype(np.int64)
    src[0] = 0                                             # a corner: most voxels outside
    tg = np.random.default_rng(n + 1).random((n, 17, 17, 17)) * 1e-3
    tg[tg < 2e-4] = 0.0                                    # 0 ln 0 = 0
    Ws, bs = so.init_params(3, noise=0.05)
    with FDiRW(shape, synth.random_diffusivity(shape, 5, 3.0), 0.1, 8, 1, "fp32") as f:
        net = Net(fdirw.pack_params(Ws, bs))
        acts, z, _, pg, loss = net.trace(f.ctx, src, tg)
        for _ in range(2):
            g2, loss2 = net.gradients(f.ctx, src, tg)
            assert np.array_equal(pg, g2) and loss == loss2
        net.close()
    inside = np.stack([a.reshape(16, 17, 17, 17)[1] for a in acts[0]]) > 0x3F00        # BF16 bits of 0.5
    zz = z.astype(np.float64).reshape(tg.shape)
    y = np.exp(zz)
    parts = [y, -tg * zz, tg * np.log(np.where(tg > 0.0, tg, 1.0)), -tg]
    want = sum(float(p[inside].sum()) for p in parts) / n
    size = sum(float(np.abs(p[inside]).sum()) for p in parts) / n
    assert abs(loss - want) <= 1e-12 * size
