"""The median of a large cube (one pass over the voxels, the keys near a
sampled bracket kept in a list) against a full sort: noise, NaN voxels,
storage types and brick sizes, half of all voxels equal (the list
overflows), a constant cube, and a cube whose sampled voxels are all
outliers (the bracket misses the median); the last three end in the passes
over all voxels.  Sizes just below and above the one from which it is used."""
import numpy as np
import pytest

from tests.helpers import cuda_or_skip

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    return cuda_or_skip()


def _noise(torch, dims):
    g = torch.Generator(device="cuda").manual_seed(5)
    return torch.randn(dims[::-1], generator=g, device="cuda") + 0.01


def _expected(torch, stored):
    v = stored.float().reshape(-1)
    v = torch.sort(v[~torch.isnan(v)]).values
    return v[(v.numel() + 1) // 2 - 1].item()


def _check(torch, cube, store="f32", brick=0):
    import paper_1211_4896_gb300 as P
    dt = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}[store]
    vol = P.Volume(cube.contiguous(), store, brick=brick)
    try:
        want = _expected(torch, cube.to(dt))
        assert P.median(vol) == want
        assert P.median(vol) == want                     # the kept scratch again
        m = P.moments(vol)
        assert m["count"] == int((~torch.isnan(cube)).sum())
    finally:
        vol.close()


@pytest.mark.parametrize("dims", [(321, 320, 326), (325, 324, 319), (340, 257, 401)])   # 2^25 lies between the first two
def test_noise(torch, dims):
    _check(torch, _noise(torch, dims))


@pytest.mark.parametrize("store,brick", [("f16", 16), ("bf16", 32), ("f32", 64)])
def test_storage_and_bricks(torch, store, brick):
    cube = _noise(torch, (337, 321, 341))
    cube.reshape(-1)[::7] = float("nan")
    _check(torch, cube, store, brick)


def test_many_equal_values_and_a_constant(torch):
    cube = _noise(torch, (330, 330, 330))
    flat = cube.reshape(-1)
    flat[flat.abs() < 0.7] = 0.0
    _check(torch, cube)
    cube.fill_(-3.5)
    _check(torch, cube)


def test_a_sample_that_misleads(torch):
    """Outliers exactly at the sampled places: voxel (x, y, z) of the brick of
    sample q at the bits of a hash of q."""
    nx, ny, nz, b = 337, 321, 341, 16
    cube = _noise(torch, (nx, ny, nz))
    nb = [-(-(n - 1) // b) for n in (nx, ny, nz)]
    q = np.arange(1 << 20, dtype=np.uint64)
    brick = (q * np.uint64(nb[0] * nb[1] * nb[2])) >> np.uint64(20)
    h = (q * np.uint64(0x9E3779B1)) & np.uint64(0xffffffff)
    h ^= h >> np.uint64(15)
    h = (h * np.uint64(0x9E3779B1)) & np.uint64(0xffffffff)
    c = [(h >> np.uint64(s)) & np.uint64(b - 1) for s in (8, 16, 24)]
    x = (brick % np.uint64(nb[0])) * np.uint64(b) + c[0]
    y = (brick // np.uint64(nb[0]) % np.uint64(nb[1])) * np.uint64(b) + c[1]
    z = (brick // np.uint64(nb[0] * nb[1])) * np.uint64(b) + c[2]
    ok = (x < nx) & (y < ny) & (z < nz)
    at = ((z * np.uint64(ny) + y) * np.uint64(nx) + x)[ok].astype(np.int64)
    cube.reshape(-1)[torch.from_numpy(at).cuda()] = 1e6
    _check(torch, cube)


@pytest.mark.parametrize("store", ["f32", "f16"])
@pytest.mark.parametrize("lo,hi,nb", [(-4.0, 4.0, 256), (-3.7, 5.3, 1000), (0.1, 0.7, 7), (-1e-3, 1e3, 16384), (0.0, 3.0, 1)])
def test_histogram_of_a_large_cube(torch, store, lo, hi, nb):
    """From 2^23 voxels on the bins near an edge are decided by the edges'
    floats: the counts of the FP64 expression, values on edges included."""
    import paper_1211_4896_gb300 as P
    cube = _noise(torch, (210, 203, 198))
    flat = cube.reshape(-1)
    edges = lo + (hi - lo) * torch.arange(nb + 1, device="cuda", dtype=torch.float64) / nb
    for k, t in enumerate((edges.float(), torch.nextafter(edges.float(), torch.full_like(edges, 9e9).float()),
                           torch.nextafter(edges.float(), torch.full_like(edges, -9e9).float()))):
        flat[k * 20000:k * 20000 + t.numel()] = t
    vol = P.Volume(cube, store)
    try:
        got = P.histogram(vol, lo, hi, nb)
        v = (cube if store == "f32" else cube.half()).double().reshape(-1).cpu().numpy()
        v = v[(v >= lo) & (v <= hi)]
        b = np.clip(np.floor((v - lo) / (hi - lo) * nb), 0, nb - 1).astype(np.int64)
        assert np.array_equal(got.cpu().numpy(), np.bincount(b, minlength=nb))
    finally:
        vol.close()
