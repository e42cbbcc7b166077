"""A sub-box's samples are found as one run per ray and marched without a test
per sample.  The runs of a partition into single-cell slabs and uneven boxes
add up to the whole render's sample counts, and the composite equals it: rays
along and across the axes (both signs, so that a run is entered through either
face), grazing rays, rays that miss, an eye inside the grid, steps from a
tenth to several voxels, every storage type."""
import pytest

import synth
from tests.helpers import cuda_or_skip

pytestmark = pytest.mark.gpu
DIMS = (19, 23, 17)
CUTS = [[0, 1, 2, 9, 17, 18], [0, 11, 22], [0, 8, 15, 16]]


@pytest.fixture(scope="module")
def torch():
    return cuda_or_skip()


def _cams():
    c = [0.5 * (d - 1) for d in DIMS]
    for f, up in (((0, 0, 1), (0, 1, 0)), ((0, 0, -1), (0, 1, 0)), ((-1, 0, 0), (0, 0, 1)), ((0, 1, 0), (1, 0, 0)),
                  ((0.6, -0.5, 0.62), (0, 1, 0)), ((-0.7, 0.1, 0.7), (0, 1, 0))):
        eye = tuple(c[a] - 60.0 * f[a] for a in range(3))
        yield synth.camera_ortho(eye, f, up, 30.0, 41, 37)
        yield synth.camera_persp(eye, f, up, 30.0, 33, 29)
    yield synth.camera_persp(tuple(c), (0.3, 0.5, -0.8), (0, 1, 0), 70.0, 31, 33)      # from inside


@pytest.mark.parametrize("store,step", [("f32", 0.1), ("f32", 0.73), ("f32", 4.1), ("f16", 0.5), ("bf16", 1.0)])
def test_runs_partition_every_ray(torch, store, step):
    import paper_1211_4896_gb300 as P
    cube = synth.hi_cube(DIMS, n_blobs=4, n_disks=0, seed=8)
    vol = P.Volume(cube.cuda(), store)
    tf = torch.from_numpy(synth.tf_random_pwl(seed=2, alpha_max=0.2)).cuda()
    boxes = [((x0, y0, z0), (x1, y1, z1)) for x0, x1 in zip(CUTS[0], CUTS[0][1:])
             for y0, y1 in zip(CUTS[1], CUTS[1][1:]) for z0, z1 in zip(CUTS[2], CUTS[2][1:])]
    try:
        for cam in _cams():
            img, ns = P.render(vol, cam, tf, -3.0, 30.0, step)
            parts = [P.render_subbox(vol, cam, tf, -3.0, 30.0, step, a, b) for a, b in boxes]
            assert torch.equal(sum(p[2] for p in parts), ns)
            for part, depth, count in parts:
                assert torch.equal(torch.isinf(depth), count == 0)
                assert torch.equal(part[..., 3] == 1.0, (part[..., :3] == 0.0).all(-1) & (part[..., 3] == 1.0))
            out = P.composite([p[0] for p in parts], [p[1] for p in parts])
            assert (out - img).abs().max().item() <= 1e-5          # the order of the products: 45 partials of 2^-24
    finally:
        vol.close()
