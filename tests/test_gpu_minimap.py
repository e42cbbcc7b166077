"""The mini-map's one-pass sums (two floats a sum) against the statistics in
64 bits: regions of one voxel, thin and ragged ones, ones larger than the
one-pass limit, brick edges, all storage types, and data that the sums hand
to the two FP64 passes (NaN, infinities, squares beyond the float range on
either side, an outlier as the shift).  The result is the 64-bit one rounded
to float, so half an ulp of a float (6e-8) is allowed, and as much again for
the sums' own error."""
import numpy as np
import pytest

from tests.helpers import cuda_or_skip

pytestmark = pytest.mark.gpu
TOL = 1.2e-7


@pytest.fixture(scope="module")
def torch():
    return cuda_or_skip()


def _reference(cube, r):
    nz, ny, nx = cube.shape
    m = [-(-n // q) for n, q in zip((nx, ny, nz), r)]
    out = np.empty((m[2], m[1], m[0], 2))
    with np.errstate(all="ignore"):
        for k in range(m[2]):
            for j in range(m[1]):
                for i in range(m[0]):
                    b = cube[k * r[2]:(k + 1) * r[2], j * r[1]:(j + 1) * r[1], i * r[0]:(i + 1) * r[0]]
                    b = b.astype(np.float64)
                    out[k, j, i] = b.mean(), b.std()
    return out


def _check(torch, cube, r, store="f32"):
    import paper_1211_4896_gb300 as P
    vol = P.Volume(torch.from_numpy(np.ascontiguousarray(cube)).cuda(), store)
    try:
        got = P.minimap(vol, r).cpu().numpy().astype(np.float64)
    finally:
        vol.close()
    dt = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}[store]
    ref = _reference(torch.from_numpy(cube).to(dt).to(torch.float32).numpy(), r)
    assert np.array_equal(np.isnan(got), np.isnan(ref))
    fin = np.isfinite(ref)
    assert np.array_equal(got[~fin & ~np.isnan(ref)], ref[~fin & ~np.isnan(ref)])
    assert np.all(np.abs(got - ref)[fin] <= TOL * np.abs(ref[fin]) + 1e-38), np.abs(got - ref)[fin].max()


@pytest.mark.parametrize("store", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("region", [(1, 1, 1), (2, 3, 5), (17, 16, 15), (40, 1, 1), (1, 1, 40), (64, 64, 64)])
def test_regions(torch, region, store):
    rng = np.random.default_rng(1)
    _check(torch, (rng.standard_normal((37, 50, 41)) + 3.0).astype(np.float32), region, store)


def test_region_beyond_the_one_pass_limit(torch):
    rng = np.random.default_rng(2)
    _check(torch, rng.standard_normal((130, 130, 130)).astype(np.float32), (130, 130, 128))


@pytest.mark.parametrize("name", ["offset", "outlier", "nan", "inf", "huge", "tiny", "constant", "mixed"])
def test_values(torch, name):
    rng = np.random.default_rng(3)
    cube = rng.standard_normal((24, 20, 33)).astype(np.float32)
    if name == "offset":
        cube = (cube * 1e-3 + 1e3).astype(np.float32)
    elif name == "outlier":
        cube[0, 0, 0] = 1e7
    elif name == "nan":
        cube[3, 4, 5] = np.nan
    elif name == "inf":
        cube[3, 4, 5], cube[20, 15, 30] = np.inf, -np.inf
    elif name == "huge":
        cube *= np.float32(1e25)
    elif name == "tiny":
        cube *= np.float32(1e-25)
    elif name == "constant":
        cube[:] = 0.1
    elif name == "mixed":
        cube[:, :, :12] = 0.0
        cube[5, 5, 20] = 3e19
    _check(torch, cube, (12, 10, 8))
