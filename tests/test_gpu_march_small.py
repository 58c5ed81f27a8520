"""Launches of the block march that do not fill every CTA with sources: each CTA takes an even share of them, warps without
a source stay out of the march, and a launch of coarse blocks that leaves one per SM at most takes one thread a column.
Bit for bit against the one-column march, for source counts around an SM's and a wave's worth (152 SMs), with whatever an
earlier kernel left in shared memory."""
import numpy as np
import pytest

from paper_2408_11376_gb300 import FDiRW, FDiRWCoarse, fdirw, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _library():
    from paper_2408_11376_gb300 import build
    build.build()


def _leave_values_in_shared_memory():
    shape = (13, 12, 11)
    D = synth.random_diffusivity(shape, 1, 3.0)
    with FDiRW(shape, D, 9 * fdirw.fdirw_stable_dt(shape, D), 8, 9, march_parts=5) as f:
        f.kernels()


@pytest.mark.parametrize("R", [1, 2, 3, 4, 5, 7, 8])
@pytest.mark.parametrize("shape", [(1, 1, 1), (19, 8, 1), (9, 17, 1), (7, 13, 11), (32, 19, 6), (41, 89, 1), (25, 20, 10),
                                   (24, 19, 14), (32, 19, 24), (17, 18, 1), (5, 61, 1)])
def test_small_launches_equal_the_column_march(R, shape):
    D = synth.random_diffusivity(shape, 20 + R, 5.0)
    dt = fdirw.fdirw_stable_dt(shape, D)
    dt = dt if np.isfinite(dt) else 1.0
    src = np.unique(np.linspace(0, D.size - 1, 600).astype(np.int64))
    out = []
    for parts in (1, 4, 0, 4):
        _leave_values_in_shared_memory()
        with FDiRW(shape, D, 7 * dt, R, 7, "bf16", march_parts=parts) as f:
            f.kernels()
            out.append(f.read_kernels(src))
            o = np.empty(D.size)
            f.step(np.arange(D.size) * 0.25 + 1.0, o)
        out[-1] = np.concatenate([out[-1].ravel(), o])
    assert all(np.array_equal(out[0], v) for v in out[1:])


@pytest.mark.parametrize("B,R,shape", [(1, 1, (13, 12, 11)), (1, 2, (31, 30, 29)), (3, 1, (18, 18, 17)), (3, 2, (60, 50, 40)),
                                       (3, 4, (30, 30, 30)), (3, 6, (25, 26, 27)), (5, 3, (31, 32, 33)), (5, 6, (40, 41, 32)),
                                       (1, 8, (9, 8, 7)), (7, 5, (41, 43, 42)), (3, 8, (19, 18, 20)), (5, 8, (33, 31, 30))])
@pytest.mark.parametrize("open_surface", [False, True])
def test_coarse_matrix_equals_the_column_march(B, R, shape, open_surface):
    """Against the same context with a velocity of zero, whose blocks always take one thread a column."""
    p = synth.sphere_packing(shape, 0.5, 5, r_range=(1.0, 2.0))
    D, liquid = synth.diffusivity_two_phase(p, 1.0, 1e-6), (~p.solid).astype(np.uint8)
    dt = 0.9 * fdirw.fdirw_stable_dt(shape, D)
    nb = int(np.prod([-(-n // B) for n in shape]))
    out = []
    for flow in (True, False, False):
        _leave_values_in_shared_memory()
        with FDiRWCoarse(shape, D, liquid, B, 6 * dt, R, 6) as f:
            if open_surface:
                f.far_field(100.0, 0.5)
            if flow:
                f.set_velocity(np.zeros(3 * D.size))
            f.kernels()
            out.append(f.read_coarse(np.arange(nb)))
    assert np.array_equal(out[0], out[1]) and np.array_equal(out[0], out[2])


@pytest.mark.parametrize("shape,n_sub", [((1, 1, 1), 2), ((1, 1, 5), 1), ((60, 1, 3), 9), ((2, 31, 2), 4), ((7, 9, 11), 30)])
def test_fp64_march_of_radius_one(shape, n_sub):
    """Every level of a column is computed there: kernels against the oracle, and the z-slabs of a streamed cache."""
    import oracle
    D = synth.random_diffusivity(shape, 60, 4.0)
    lam = oracle.stable_dt_sub(shape, D)
    lam = lam if np.isfinite(lam) else 1.0
    src, c = np.arange(D.size), synth.random_field(D.size, 61)
    out = []
    with FDiRW(shape, D, n_sub * lam, 1, n_sub, "fp64") as f:
        f.kernels()
        ks = f.read_kernels(src).reshape(D.size, -1)
        fixed = f.info()["device_bytes"] - f.info()["cache_bytes"] - D.size * (8 + 8 * 27)
    ref = oracle.kernels(shape, D, lam, 1, n_sub, src)[0].reshape(D.size, -1)
    assert (np.linalg.norm(ks - ref, axis=1) / np.linalg.norm(ref, axis=1)).max() <= 1e-13
    # one z plane of the cache at a time, then all of it
    for limit in ([fixed + 8 * D.size + 27 * 8 * shape[0] * shape[1]] if shape[2] > 1 else []) + [0]:
        with FDiRW(shape, D, n_sub * lam, 1, n_sub, "fp64", mem_limit=limit) as f:
            out.append(np.empty(D.size))
            f.step(c, out[-1], 2)
            assert f.info()["n_chunks"] == (shape[2] if limit else 1)
    assert all(np.array_equal(out[-1], o) for o in out)
