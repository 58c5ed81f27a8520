"""The superposition's row groups, padded cache rows and packed arithmetic where they can go wrong: rows of one vector
and less, rows that end inside a vector, every radius class, every storage type, the largest and the smallest grids of
a block, against the same gather in float64 on the kernels that the library stored (read back exactly)."""
import numpy as np
import pytest
import torch

from paper_2408_11376_gb300 import FDiRW, FDiRWBatch, fdirw, synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
# Relative to sum |terms|: float-float keeps about 2^-44 of it over 9261 terms; FP32 rows are off by at most
# (2R+1) 2^-24 each (21 terms), and the mass restoration moves a value by no more than the total of that.
TOL = {"ff": 2.0 ** -44, "fp32": 2 * 22 * 2.0 ** -24, "fp64": 9261 * 2.0 ** -53}


@pytest.fixture(scope="module", autouse=True)
def _library():
    from paper_2408_11376_gb300 import build
    build.build()


def _superpose(shape, ks, c):
    """sum over sources of c(s) k_s in float64; ks [N, W, W, W]."""
    nx, ny, nz = shape
    W = ks.shape[1]
    R = W // 2
    out = np.zeros((nz + 2 * R, ny + 2 * R, nx + 2 * R))
    for s in range(nx * ny * nz):
        x, y, z = s % nx, (s // nx) % ny, s // (nx * ny)
        out[z:z + W, y:y + W, x:x + W] += c[s] * ks[s]
    return out[R:R + nz, R:R + ny, R:R + nx].reshape(-1)


@pytest.mark.parametrize("prec,accum", [("fp32", "ff"), ("bf16", "ff"), ("fp16", "fp32"), ("bf16", "fp32"), ("fp32", "fp32"),
                                        ("fp64", "ff")])
@pytest.mark.parametrize("shape,R", [((1, 3, 9), 1), ((7, 5, 3), 2), ((9, 4, 5), 3), ((8, 5, 4), 4), ((23, 6, 5), 8),
                                     ((17, 9, 3), 7), ((16, 9, 5), 10), ((33, 5, 7), 2)])
def test_gather_matches_its_stored_kernels(prec, accum, shape, R):
    if prec == "fp64" and R > 8:
        pytest.skip("the FP64 path takes R <= 8")
    N = int(np.prod(shape))
    D = synth.random_diffusivity(shape, 3 + R, 3.0)
    dt = fdirw.fdirw_stable_dt(shape, D)
    c0 = synth.random_field(N, 4, -1.0, 2.0)
    with FDiRW(shape, D, 5 * dt, R, 5, prec, accum=accum) as f:
        out = np.empty(N)
        f.step(c0, out, 1)
        ks = f.read_kernels(np.arange(N))
    ref = _superpose(shape, ks, c0)
    size = _superpose(shape, np.abs(ks), np.abs(c0))
    tol = TOL["fp64" if prec == "fp64" else accum] * (size if accum == "ff" else size.max())
    assert np.all(np.abs(out - ref) <= tol), np.max(np.abs(out - ref) / tol)


@pytest.mark.parametrize("accum", ["ff", "fp32"])
def test_batch_of_ragged_structures_equals_each_alone(accum):
    shapes, R = [(9, 6, 5), (16, 4, 3), (21, 3, 4)], 4
    Ds = [synth.random_diffusivity(s, 90 + i, 2.0) for i, s in enumerate(shapes)]
    dt = min(fdirw.fdirw_stable_dt(s, d) for s, d in zip(shapes, Ds))
    c0 = [synth.random_field(int(np.prod(s)), 95 + i) for i, s in enumerate(shapes)]
    alone = []
    for s, d, c in zip(shapes, Ds, c0):
        out = np.empty_like(c)
        with FDiRW(s, d, 6 * dt, R, 6, "bf16", accum=accum) as f:
            f.step(c, out, 1)
        alone.append(out)
    got = np.empty(sum(c.size for c in c0))
    with FDiRWBatch(shapes, Ds, 6 * dt, R, R, 6, "bf16", accum=accum) as f:
        f.step(np.concatenate(c0), got, 1)
    # FP32 sums: the batch restores each structure's mass with sums in another order (FP64 rounding)
    assert np.max(np.abs(got - np.concatenate(alone))) <= (0.0 if accum == "ff" else 1e-13)
