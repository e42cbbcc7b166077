"""Sparse views and views that cover few pixels march eight lanes to a ray: images and sample counts bit for
bit those of the staged march (one ray to a lane), for rays of fewer samples
than lanes and of many, image edges that cut the 2 x 2 tiles, early
termination at every place in a round, opaque and transparent tables, all
storage types and brick sizes (bricks, row copies and blocked copies;
texture layers and paired copies)."""
import pytest

import synth
from tests.helpers import cuda_or_skip

pytestmark = pytest.mark.gpu
DIMS = (50, 43, 61)


@pytest.fixture(scope="module")
def torch():
    return cuda_or_skip()


@pytest.mark.parametrize("store,brick", [("f32", 16), ("f32", 64), ("f16", 16), ("bf16", 32), ("f16", 64)])
def test_groups_match_single_lanes(torch, store, brick):
    import paper_1211_4896_gb300 as P
    from paper_1211_4896_gb300 import _lib as L
    vol = P.Volume(synth.hi_cube(DIMS, n_blobs=9, n_disks=0, seed=4).cuda(), store, brick=brick)
    tables = [torch.from_numpy(t).cuda() for t in (synth.tf_ramp(256), synth.tf_random_pwl(seed=6, alpha_max=0.5))]
    c = [0.5 * (d - 1) for d in DIMS]
    try:
        for q, (f, up) in enumerate((((0, 0, 1), (0, 1, 0)), ((1, 0, 0), (0, 1, 0)), ((0, -1, 0), (1, 0, 0)),
                                     ((0.6, -0.5, 0.62), (0, 1, 0)))):
            eye = tuple(c[a] - 150.0 * f[a] for a in range(3))
            w, h = ((13, 9), (8, 11), (15, 14), (1, 2))[q]
            for cam in (synth.camera_ortho(eye, f, up, 70.0, w, h), synth.camera_persp(eye, f, up, 30.0, w, h)):
                for step, ert in ((0.31, 2.0), (0.5, 0.6), (0.5, 0.99), (9.0, 2.0), (40.0, 0.3)):
                    for tf in tables:
                        a, na = P.render(vol, cam, tf, -3.0, 30.0, step, ert)
                        b, nb = P.render(vol, cam, tf, -3.0, 30.0, step, ert, filter=L.VR_FILTER_SOFTWARE_STAGED)
                        assert torch.equal(na, nb) and torch.equal(a, b)
    finally:
        vol.close()


@pytest.mark.parametrize("store", ["f32", "f16", "bf16"])
def test_small_dense_views(torch, store):
    """Dense views of a few hundred tiles: texture layers (float) and paired
    copies; the oblique one leaves part of the image uncovered, the last has
    the eye inside the volume."""
    import paper_1211_4896_gb300 as P
    from paper_1211_4896_gb300 import _lib as L
    vol = P.Volume(synth.hi_cube(DIMS, n_blobs=9, n_disks=0, seed=4).cuda(), store)
    tables = [torch.from_numpy(t).cuda() for t in (synth.tf_ramp(256), synth.tf_random_pwl(seed=6, alpha_max=0.5))]
    c = [0.5 * (d - 1) for d in DIMS]
    try:
        cams = [synth.camera_ortho((c[0], c[1], -50.0), (0, 0, 1), (0, 1, 0), 42.0, 61, 47),
                synth.camera_persp((c[0] - 150.0, c[1], c[2]), (1, 0, 0), (0, 0, 1), 30.0, 90, 77),
                synth.camera_random_persp(DIMS, seed=3, width=131, height=90),
                synth.camera_persp(tuple(c), (0.3, 0.5, -0.8), (0, 1, 0), 70.0, 65, 66)]
        for cam in cams:
            for step, ert in ((0.31, 2.0), (0.5, 0.6), (1.0, 0.99)):
                for tf in tables:
                    a, na = P.render(vol, cam, tf, -3.0, 30.0, step, ert)
                    b, nb = P.render(vol, cam, tf, -3.0, 30.0, step, ert, filter=L.VR_FILTER_SOFTWARE_STAGED)
                    assert torch.equal(na, nb) and torch.equal(a, b)
    finally:
        vol.close()


@pytest.mark.parametrize("store", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("view", range(3))
def test_a_cut_of_an_image_marched_in_groups(torch, store, view):
    """The middle 64 x 64 pixels of a 256 x 256 orthographic image (which has a
    ray to a lane) are, bit for bit, the 64 x 64 image of the same rays (eight
    lanes to a ray): composite, maximum, sigma clipping, a sub-box."""
    import paper_1211_4896_gb300 as P
    vol = P.Volume(synth.hi_cube(DIMS, n_blobs=9, n_disks=0, seed=4).cuda(), store)
    c = [0.5 * (d - 1) for d in DIMS]
    f, up = (((0, 0, 1), (0, 1, 0)), ((-1, 0, 0), (0, 0, 1)), ((0.6, -0.5, 0.62), (0, 1, 0)))[view]
    eye = tuple(c[a] - 150.0 * f[a] for a in range(3))
    big = synth.camera_ortho(eye, f, up, 40.0, 256, 256)
    cut = synth.camera_ortho(eye, f, up, 10.0, 64, 64)
    at = slice(96, 160)
    mm = P.minimap(vol, (9, 8, 7))
    kw = dict(mode=P.VR_MODE_SIGMA, minimap=mm, region=(9, 8, 7))
    try:
        for tf in [torch.from_numpy(t).cuda() for t in (synth.tf_ramp(256), synth.tf_random_pwl(seed=6, alpha_max=0.5))]:
            for step, ert in ((0.31, 2.0), (0.7, 0.9)):
                calls = [lambda cam: P.render(vol, cam, tf, -3.0, 30.0, step, ert),
                         lambda cam: P.render(vol, cam, tf, -3.0, 30.0, step, mode=P.VR_MODE_MIP),
                         lambda cam: P.render(vol, cam, tf, 0.0, 8.0, step, ert, **kw),
                         lambda cam: P.render_subbox(vol, cam, tf, -3.0, 30.0, step, (3, 5, 7), (40, 31, 52))]
                for call in calls:
                    for a, b in zip(call(big), call(cut)):
                        assert torch.equal(a[at, at], b)
    finally:
        vol.close()
