"""Sigma clipping with a caller's mini-map of more than 2^31 points (regions of
one voxel): rays beside the points past 2^31 give the image of the same rays
through a small cut of the volume with its cut of the map.  Values vary along
x alone and every position is exact in 32 bits, so the images differ by
rounding at most."""
import pytest

from tests.helpers import cuda_or_skip

pytestmark = pytest.mark.gpu

NX, NY, NZ = 2048, 1024, 1030                 # point (0, 0, 1024) is number 2^31
Y0, Z0, NYC, NZC = 497, 1020, 8, 10           # the cut


@pytest.fixture(scope="module")
def volumes():
    torch = cuda_or_skip()
    if torch.cuda.mem_get_info()[0] < (60 << 30):
        pytest.skip("needs 60 GB of device memory")
    import paper_1211_4896_gb300 as P
    line = (3.0 * torch.sin(torch.arange(NX, device="cuda") * 0.2)).half()

    def make(ny, nz, z0):
        vol = P.Volume(line.expand(nz, ny, NX).contiguous(), "f16")
        mm = torch.zeros((nz, ny, NX, 2), device="cuda")
        mm[..., 1] = 1.0
        mm[max(0, 1024 - z0):, ..., 0] = 1.0
        mm[max(0, 1024 - z0):, ..., 1] = 0.5
        return vol, mm
    big, small = make(NY, NZ, 0), make(NYC, NZC, Z0)
    yield big, small
    big[0].close()
    small[0].close()


@pytest.mark.parametrize("w,h", [(6, 4), (320, 256)])        # the cut: eight lanes to a ray, a lane to a ray
def test_points_past_two_to_the_31(volumes, w, h):
    import torch
    import paper_1211_4896_gb300 as P
    t = torch.linspace(0.0, 1.0, 64, device="cuda")
    tf = torch.stack([t, 1.0 - t, t * t, 0.02 * t], 1).contiguous()

    def image(vm, y, z):
        vol, mm = vm
        cam = dict(kind=P.VR_CAMERA_ORTHO, eye=(-10.0, y, z), forward=(1.0, 0.0, 0.0), up=(0.0, 1.0, 0.0),
                   fov_y_deg=0.0, ortho_height=4.0, width=w, height=h)
        return P.render(vol, cam, tf, -4.0, 6.0, 1.0, 2.0, mode=P.VR_MODE_SIGMA, minimap=mm, region=(1, 1, 1))
    big, nb = image(volumes[0], 500.0, 1026.0)
    small, ns = image(volumes[1], 500.0 - Y0, 1026.0 - Z0)
    assert int(nb.min()) == 2047 and torch.equal(nb, ns)
    assert (big - small).abs().max().item() <= 1e-5
    assert big.std().item() > 0.01
