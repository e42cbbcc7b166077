"""Histogram bins whose edge falls at or near zero, in a cube large enough for
the edges' floats: floats lie far closer together there than anywhere else in
the range, and the FP64 expression that decides a bin changes its mind at
1e-17 or so rather than at the float nearest to the edge.  Counts are whole
numbers and equal those of the expression."""
import numpy as np
import pytest

from tests.helpers import cuda_or_skip

pytestmark = pytest.mark.gpu

NEAR_ZERO = [0.0, -0.0] + [s * v for s in (1.0, -1.0)
                           for v in (1e-45, 1e-40, 1.2e-38, 1e-30, 1e-20, 1e-18, 1e-17, 5.5e-17, 5.6e-17, 1e-16, 1e-15, 1e-12)]


@pytest.fixture(scope="module")
def cube():
    torch = cuda_or_skip()
    g = torch.Generator(device="cuda").manual_seed(9)
    c = torch.randn((198, 203, 210), generator=g, device="cuda")
    flat = c.reshape(-1)
    for q, v in enumerate(NEAR_ZERO):
        flat[q * 1000:q * 1000 + 100 + q] = v
    flat[7000000:7500000] = 0.0                      # a blanked part
    return c


@pytest.mark.parametrize("lo,hi,nb", [
    (-0.1, 0.2, 30), (-1.7, 1.5, 256), (-1.0, 1.0, 256), (-3.9, 2.5, 128), (-1.3, 2.6, 300), (-0.01, 0.05, 60),
    (-0.05, 0.1, 30), (-0.2, 0.4, 60), (-0.4, 0.8, 120), (0.0, 1.0, 64), (-1.0, 0.0, 64), (-1e-30, 3.0, 100),
    (-4.0, 4.0, 2), (-4.0, 4.0, 16384)])
def test_edges_near_zero(cube, lo, hi, nb):
    import paper_1211_4896_gb300 as P
    vol = P.Volume(cube, "f32")
    try:
        got = P.histogram(vol, lo, hi, nb).cpu().numpy()
    finally:
        vol.close()
    v = cube.double().reshape(-1).cpu().numpy()
    v = v[(v >= lo) & (v <= hi)]
    b = np.clip(np.floor((v - lo) / (hi - lo) * nb), 0, nb - 1).astype(np.int64)
    assert np.array_equal(got, np.bincount(b, minlength=nb))


def test_no_scratch_where_the_edges_are_not_used():
    """A small volume's histogram makes no device allocation: the failure armed
    before it is left to the next call that makes one."""
    torch = cuda_or_skip()
    import paper_1211_4896_gb300 as P
    from paper_1211_4896_gb300 import _lib as L
    c = torch.randn((30, 40, 50), device="cuda")
    vol = P.Volume(c, "f32")
    try:
        L.vr_debug_fail_alloc(0)
        got = P.histogram(vol, -1.0, 1.0, 10)
        with pytest.raises(L.VRError) as e:
            P.moments(vol)
        assert e.value.status == L.VR_ERR_OOM
        assert int(got.sum()) == int((c.abs() <= 1.0).sum())
    finally:
        L.vr_debug_fail_alloc(-1)
        vol.close()
