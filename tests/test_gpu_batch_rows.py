"""Cache rows of a batch at a memory limit between its packed and its padded kernels, and with a structure narrower than
a vector: one chunk, readable kernels and the fields of each structure alone, bit for bit."""
import numpy as np
import pytest

from paper_2408_11376_gb300 import FDiRW, FDiRWBatch, fdirw, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _library():
    from paper_2408_11376_gb300 import build
    build.build()


def _alone(shapes, Ds, dt, R, n_sub, prec, cs):
    out = []
    for s, d, c in zip(shapes, Ds, cs):
        o = np.empty_like(c)
        with FDiRW(s, d, n_sub * dt, R, n_sub, prec) as f:
            f.step(c, o, 2)
        out.append(o)
    return np.concatenate(out)


@pytest.mark.parametrize("prec", ["fp32", "bf16"])
@pytest.mark.parametrize("shapes", [[(17, 6, 5)] * 3, [(9, 7, 6), (33, 5, 4)], [(5, 6, 7), (16, 5, 4), (21, 4, 6)]])
def test_batch_rows(shapes, prec):
    R, n_sub, n = 4, 6, len(shapes)
    Ds = [synth.random_diffusivity(s, 30 + i, 2.0) for i, s in enumerate(shapes)]
    dt = min(fdirw.fdirw_stable_dt(s, d) for s, d in zip(shapes, Ds))
    cs = [synth.random_field(int(np.prod(s)), 40 + i) for i, s in enumerate(shapes)]
    c, want = np.concatenate(cs), _alone(shapes, Ds, dt, R, n_sub, prec, cs)
    packed = 729 * (4 if prec == "fp32" else 2) * sum((x.size + 15) // 16 * 16 for x in cs)
    with FDiRWBatch(shapes, Ds, n_sub * dt, R, R, n_sub, prec) as f:
        got = np.empty_like(c)
        f.step(c, got, 2)
        assert np.array_equal(got, want)
        ks = f.read_kernels(np.arange(c.size))
        i = f.info()
        fixed = i["device_bytes"] - i["cache_bytes"] - c.size * (8 + 8 * 729)
    # room for the packed kernels and for reading one of them back, and for no more
    with FDiRWBatch(shapes, Ds, n_sub * dt, R, R, n_sub, prec, mem_limit=fixed + packed + 11 * 256 + 8 + 8 * 729) as f:
        f.step(c, got, 2)
        assert f.info()["n_chunks"] == 1 and np.array_equal(got, want)
        assert np.array_equal(f.read_kernels([c.size - 1]), ks[-1:])
