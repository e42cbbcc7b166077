"""The median of large cubes with many equal values near the middle, which the
list of the one-pass median cannot hold (blanked, integer and 16-bit cubes),
and of one whose sampled voxels are outliers of distinct values (a bracket
that misses the median): the value of the sorted cube's rank."""
import numpy as np
import pytest

from tests.helpers import cuda_or_skip

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    return cuda_or_skip()


def _check(torch, cube, store="f32"):
    import paper_1211_4896_gb300 as P
    dt = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}[store]
    v = cube.to(dt).float().reshape(-1)
    v = torch.sort(v[~torch.isnan(v)]).values
    want = v[(v.numel() + 1) // 2 - 1].item() if v.numel() else float("nan")
    vol = P.Volume(cube.contiguous(), store)
    try:
        got = P.median(vol)
    finally:
        vol.close()
    assert got == want or (np.isnan(got) and np.isnan(want))


def _noise(torch, dims=(331, 322, 340)):
    g = torch.Generator(device="cuda").manual_seed(6)
    return torch.randn(dims[::-1], generator=g, device="cuda")


@pytest.mark.parametrize("share", [0.001, 0.004, 0.0078, 0.012, 0.03, 0.6])     # the list holds 1/128
def test_share_of_equal_values(torch, share):
    cube = _noise(torch)
    n = int(cube.numel() * share)
    at = torch.randperm(cube.numel(), generator=torch.Generator(device="cuda").manual_seed(1), device="cuda")[:n]
    cube.reshape(-1)[at] = 0.0
    _check(torch, cube)


@pytest.mark.parametrize("store", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("name", ["integers", "far from zero", "constant", "half blanked", "nearly all blanked", "all blanked"])
def test_data(torch, name, store):
    cube = _noise(torch)
    if name == "integers":
        cube = torch.round(2.0 * cube)
    elif name == "far from zero":
        cube += 1000.0
    elif name == "constant":
        cube.fill_(-2.5)
    elif name == "half blanked":
        cube[:170] = float("nan")
    elif name == "nearly all blanked":
        cube.reshape(-1)[1000:] = float("nan")
    else:
        cube.fill_(float("nan"))
    _check(torch, cube, store)


def test_a_bracket_that_misses(torch):
    """Distinct outliers exactly at the sampled places: voxel (x, y, z) of the
    brick of sample q at the bits of a hash of q."""
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
    at = np.unique(((z * np.uint64(ny) + y) * np.uint64(nx) + x)[ok].astype(np.int64))
    outliers = torch.linspace(1e3, 1e6, len(at), dtype=torch.float64).float().cuda()
    cube.reshape(-1)[torch.from_numpy(at).cuda()] = outliers
    _check(torch, cube)
