"""The marches leave out the table lookup of samples below the table's leading
run of zero opacities.  Every such image equals, bit for bit, that of the
staged march (VR_FILTER_SOFTWARE_STAGED), which looks every sample up: runs of
0, 1, 2, K - 1 and K entries, a run that begins later, colours that are not
finite, an early termination that ends a ray at its first sample."""
import numpy as np
import pytest

import synth
from tests.helpers import cuda_or_skip

pytestmark = pytest.mark.gpu
K = 37


@pytest.fixture(scope="module")
def torch():
    return cuda_or_skip()


def _table(run, start=0):
    tf = synth.tf_random_pwl(seed=11, K=K, alpha_max=0.3)
    tf[:, 3] = np.maximum(tf[:, 3], 0.01)
    tf[start:start + run, 3] = 0.0
    return tf


def _tables():
    for run in (0, 1, 2, 17, K - 1, K):
        yield "run%d" % run, _table(run), 2.0
    yield "later", _table(9, start=5), 2.0
    for bad in (np.inf, np.nan):
        tf = _table(12)
        tf[3, 1] = bad
        yield "colour %r" % bad, tf, 2.0
    yield "stops at once", _table(12), 1e-9
    yield "stops early", _table(12), 0.4


@pytest.mark.parametrize("store", ["f32", "f16"])
@pytest.mark.parametrize("name,tf_np,ert", list(_tables()), ids=[t[0] for t in _tables()])
def test_transparent_run_is_exact(torch, store, name, tf_np, ert, monkeypatch):
    import paper_1211_4896_gb300 as P
    from paper_1211_4896_gb300 import _lib as L
    monkeypatch.setenv("VR_TEX_LAYERS", "0")            # the brick layouts
    dims = (29, 33, 21)
    cube = synth.hi_cube(dims, n_blobs=5, n_disks=0, seed=3)
    vol = P.Volume(cube.cuda(), store)
    tf = torch.from_numpy(tf_np).cuda()
    try:
        for size in ((40, 37), (7, 5)):                  # dense and sparse rays
            cam = synth.camera_random_persp(dims, seed=9, width=size[0], height=size[1])
            a, na = P.render(vol, cam, tf, -3.0, 30.0, 0.5, ert)
            b, nb = P.render(vol, cam, tf, -3.0, 30.0, 0.5, ert, filter=L.VR_FILTER_SOFTWARE_STAGED)
            torch.cuda.synchronize()
            assert torch.equal(na, nb)
            assert torch.equal(torch.isnan(a), torch.isnan(b))
            assert torch.equal(torch.nan_to_num(a), torch.nan_to_num(b))
            if ert == 1e-9:
                assert int(na.max()) == 1
    finally:
        vol.close()
