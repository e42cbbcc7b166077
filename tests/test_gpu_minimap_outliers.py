"""The mini-map of regions whose first voxel is far from the rest (the shift
of its sums), up to the largest region of the one-pass sums: mean and
deviation are the 64-bit ones rounded to float (6e-8), and as much again is
allowed for the sums' own error."""
import numpy as np
import pytest

from tests.helpers import cuda_or_skip

pytestmark = pytest.mark.gpu
TOL = 1.2e-7


@pytest.fixture(scope="module")
def torch():
    return cuda_or_skip()


def _check(torch, cube, region):
    import paper_1211_4896_gb300 as P
    vol = P.Volume(torch.from_numpy(np.ascontiguousarray(cube)).cuda(), "f32")
    try:
        got = P.minimap(vol, region).cpu().numpy().astype(np.float64)
    finally:
        vol.close()
    for k in range(got.shape[0]):
        for j in range(got.shape[1]):
            for i in range(got.shape[2]):
                b = cube[tuple(slice(q * r, (q + 1) * r) for q, r in zip((k, j, i), region[::-1]))].astype(np.longdouble)
                mean = b.mean()
                want = float(mean), float(np.sqrt(((b - mean) ** 2).mean()))
                assert np.all(np.abs(got[k, j, i] - want) <= TOL * np.abs(want)), (got[k, j, i], want)


@pytest.mark.parametrize("first", [0.0, 40.0, 1e5, 1e7, -1e12])
@pytest.mark.parametrize("region", [(128, 128, 128), (64, 64, 64), (128, 1, 1), (1, 3, 128), (31, 33, 32)])
def test_first_voxel_far_from_the_rest(torch, region, first):
    rng = np.random.default_rng(4)
    cube = rng.standard_normal((128, 128, 128)).astype(np.float32)
    cube[::region[2], ::region[1], ::region[0]] += np.float32(first)
    _check(torch, cube[:2 * region[2], :2 * region[1], :2 * region[0]], region)


@pytest.mark.parametrize("name", ["two values", "mostly one value", "far from zero", "1e-24", "1e24"])
def test_other_data(torch, name):
    """Quantised data, whose rounding errors do not average out, and units that
    put the squares beyond the float range."""
    rng = np.random.default_rng(5)
    cube = rng.standard_normal((128, 128, 128)).astype(np.float32)
    if name == "two values":
        cube = np.where(cube > 0.5, np.float32(0.1), np.float32(0.0))
    elif name == "mostly one value":
        cube = np.where(cube > 3.0, np.float32(0.1), np.float32(0.8))
    elif name == "far from zero":
        cube = (cube * np.float32(1e-2) + np.float32(1e3)).astype(np.float32)
    elif name == "1e-24":
        cube *= np.float32(1e-24)
    elif name == "1e24":
        cube *= np.float32(1e24)
    _check(torch, cube, (128, 128, 128))
    _check(torch, cube[:70], (50, 64, 33))
