"""Views marched in groups hand out 2 x 2 tiles only around the volume and
clear the rest of the image in blocks.  Every pixel equals that of the march
with a ray to a lane, bit for bit, in images that the volume fills, crosses,
touches at an edge or misses: volumes off every side, far away, zoomed in on,
seen from inside and edge on; odd sizes; spacings that differ by axis;
composite, maximum, sigma clipping, sub-boxes and sub-cubes of a larger grid;
sparse views in a batch."""
import pytest

import synth
from tests.helpers import cuda_or_skip

pytestmark = pytest.mark.gpu
DIMS = (21, 34, 27)


@pytest.fixture(scope="module")
def torch():
    return cuda_or_skip()


def _cams(dims, spacing=(1.0, 1.0, 1.0), origin=(0.0, 0.0, 0.0)):
    c = [o + 0.5 * (d - 1) * s for o, d, s in zip(origin, dims, spacing)]
    r = 0.5 * max((d - 1) * s for d, s in zip(dims, spacing))
    for q, (f, up) in enumerate((((0, 0, 1), (0, 1, 0)), ((1, 0, 0), (0, 0, 1)), ((0.6, -0.5, 0.62), (0, 1, 0)),
                                 ((-0.02, -1, 0.01), (0, 0, 1)))):
        w, h = ((67, 45), (130, 9), (33, 128), (101, 77))[q]
        for height, shift in ((2.5, 0.0), (9.0, 0.0), (200.0, 0.0), (0.1, 0.0), (6.0, 3.2), (6.0, -3.0), (6.0, 9.0)):
            right = [f[1] * up[2] - f[2] * up[1], f[2] * up[0] - f[0] * up[2], f[0] * up[1] - f[1] * up[0]]
            eye = [c[a] - 40.0 * r * f[a] + shift * r * (right[a] + 0.4 * up[a]) for a in range(3)]
            yield synth.camera_ortho(eye, f, up, height * r, w, h)
            yield synth.camera_persp(eye, f, up, 0.7 * height if height < 100 else 150.0, h + 2, w)
    yield synth.camera_persp(c, (0.3, 0.5, -0.8), (0, 1, 0), 70.0, 61, 33)
    yield synth.camera_persp([c[0] + 1.2 * r, c[1], c[2]], (0.05, 0.1, -1.0), (0, 1, 0), 100.0, 61, 33)


def _same(torch, monkeypatch, call):
    got = []
    for g in ("0", "1"):
        monkeypatch.setenv("VR_GROUPS", g)
        got.append(call())
    for a, b in zip(*got):
        assert torch.equal(a, b)
    return got[1]


@pytest.mark.parametrize("store,spacing", [("f32", (1.0, 1.0, 1.0)), ("f16", (0.3, 2.0, 1.0))])
def test_every_pixel(torch, monkeypatch, store, spacing):
    import paper_1211_4896_gb300 as P
    origin = (5.0, -300.0, 0.25)
    vol = P.Volume(synth.hi_cube(DIMS, n_blobs=5, n_disks=0, seed=2).cuda(), store, origin=origin, spacing=spacing)
    tf = torch.from_numpy(synth.tf_random_pwl(seed=3, alpha_max=0.4)).cuda()
    mm = P.minimap(vol, (5, 6, 7))
    bg = (0.2, 0.4, 0.6, 0.3)
    seen = 0
    try:
        for cam in _cams(DIMS, spacing, origin):
            img, ns = _same(torch, monkeypatch, lambda: P.render(vol, cam, tf, -3.0, 30.0, 0.4, 0.97, bg))
            seen += int(ns.max()) > 0
            _same(torch, monkeypatch, lambda: P.render(vol, cam, tf, -3.0, 30.0, 0.4, bg=bg, mode=P.VR_MODE_MIP))
            _same(torch, monkeypatch, lambda: P.render(vol, cam, tf, 0.0, 8.0, 0.4, bg=bg, mode=P.VR_MODE_SIGMA, minimap=mm,
                                                       region=(5, 6, 7)))
            _same(torch, monkeypatch, lambda: P.render_subbox(vol, cam, tf, -3.0, 30.0, 0.4, (3, 5, 7), (18, 30, 20)))
    finally:
        vol.close()
    assert seen > 30


def test_sub_cubes_of_a_grid(torch, monkeypatch):
    import paper_1211_4896_gb300 as P
    cube = synth.hi_cube(DIMS, n_blobs=5, n_disks=0, seed=2).cuda()
    tf = torch.from_numpy(synth.tf_random_pwl(seed=3, alpha_max=0.4)).cuda()
    off, dims = (4, 9, 12), (12, 20, 10)
    part = cube[off[2]:off[2] + dims[2], off[1]:off[1] + dims[1], off[0]:off[0] + dims[0]].contiguous()
    vol = P.Volume(part, "f32", origin=tuple(float(o) for o in off))
    lo, hi = (5, 9, 12), (15, 28, 21)
    try:
        for cam in _cams(DIMS):
            _same(torch, monkeypatch, lambda: P.render_subbox(vol, cam, tf, -3.0, 30.0, 0.4, lo, hi, global_dims=DIMS,
                                                              offset=off))
    finally:
        vol.close()


@pytest.mark.parametrize("store", ["f32", "f16"])
def test_sparse_views_of_a_batch(torch, monkeypatch, store):
    import paper_1211_4896_gb300 as P
    from paper_1211_4896_gb300 import _lib as L
    monkeypatch.delenv("VR_GROUPS", raising=False)
    dims = (90, 70, 110)
    vol = P.Volume(synth.hi_cube(dims, n_blobs=9, n_disks=0, seed=4).cuda(), store)
    tf = torch.from_numpy(synth.tf_random_pwl(seed=6, alpha_max=0.5)).cuda()
    jobs = []
    for q, h in enumerate((8, 13, 20, 5)):
        cam = synth.camera_ortho((45.0 + 30.0 * q, 35.0, -400.0 - q), (0.1 * q, 0.05, 1.0), (0, 1, 0), 4.0 * h, 90, h)
        jobs.append(dict(vol=vol, cam=cam, tf=tf, vmin=-3.0, vmax=30.0, step=0.5, ert=0.99,
                         out=torch.empty((h, 90, 4), device="cuda"),
                         nsamples=torch.empty((h, 90), device="cuda", dtype=torch.int32)))
    try:
        cj = P.render_batched(jobs)
        kept = [(j["out"].clone(), j["nsamples"].clone()) for j in jobs]
        for j in jobs:
            j["out"].zero_()
        L.vr_render_batched_noalloc(cj, 0, 0, torch.cuda.current_stream().cuda_stream)
        for j, (img, ns) in zip(jobs, kept):
            assert torch.equal(j["out"], img) and torch.equal(j["nsamples"], ns)
        for j in jobs:
            a, na = P.render(vol, j["cam"], tf, -3.0, 30.0, 0.5, 0.99, filter=L.VR_FILTER_SOFTWARE_STAGED)
            assert torch.equal(a, j["out"]) and torch.equal(na, j["nsamples"])
    finally:
        vol.close()


@pytest.mark.parametrize("store", ["f32", "f16"])
@pytest.mark.parametrize("size", [100, 111, 150, 190, 205])       # 80 and 256 covered pixels an SM of 152 lie between them
def test_the_march_that_the_table_picks(torch, monkeypatch, store, size):
    """Views between the two limits, whose kernel marches in groups or with a
    ray to a lane by the table: no leading zero opacities, one (not enough to
    leave out a sample), two, most."""
    import paper_1211_4896_gb300 as P
    vol = P.Volume(synth.hi_cube(DIMS, n_blobs=5, n_disks=0, seed=2).cuda(), store)
    mm = P.minimap(vol, (5, 6, 7))
    cams = [synth.camera_ortho((10.0, 16.5, -60.0), (0, 0, 1), (0, 1, 0), 18.0, size, size - 1),
            synth.camera_persp((80.0, -50.0, 90.0), (-0.62, 0.6, -0.7), (0, 1, 0), 12.0, size + 3, size)]
    try:
        for run in (0, 1, 2, 200):
            tab = synth.tf_random_pwl(seed=3, K=256, alpha_max=0.4)
            tab[:, 3] += 0.01
            tab[:run, 3] = 0.0
            tf = torch.from_numpy(tab).cuda()
            for cam in cams:
                calls = [lambda: P.render(vol, cam, tf, -3.0, 30.0, 0.4, 0.97),
                         lambda: P.render(vol, cam, tf, -3.0, 30.0, 0.4, mode=P.VR_MODE_MIP),
                         lambda: P.render(vol, cam, tf, 0.0, 8.0, 0.4, 0.97, mode=P.VR_MODE_SIGMA, minimap=mm, region=(5, 6, 7)),
                         lambda: P.render_subbox(vol, cam, tf, -3.0, 30.0, 0.4, (3, 5, 7), (18, 30, 20))]
                for call in calls:
                    monkeypatch.setenv("VR_GROUPS", "0")
                    a = call()
                    monkeypatch.delenv("VR_GROUPS")
                    for x, y in zip(a, call()):
                        assert torch.equal(x, y)
    finally:
        vol.close()
