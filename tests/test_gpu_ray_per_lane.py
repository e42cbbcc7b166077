"""The small images of the other tests, which march with eight lanes to a ray,
once more with a ray to a lane (VR_GROUPS=0), as full-size views are marched:
the forward against the oracle, transparent runs, maximum, sigma clipping and
sort-last, whole and by sub-boxes."""
import os
import subprocess
import sys

import pytest

from tests.helpers import cuda_or_skip
from tests.test_gpu_forward import P, torch  # noqa: F401
from tests.test_gpu_forward import (test_all_rays_miss_give_background, test_anisotropic_spacing_and_origin,  # noqa: F401
                                    test_eye_inside_volume_and_tiny_images, test_half_storage_exact_path_and_error,
                                    test_minimal_cube_and_axis_parallel_rays, test_random_views_ragged,
                                    test_staged_and_brick_paths_are_bit_identical)
from tests.test_gpu_modes import (test_mip_half_storage_on_the_rounded_cube, test_mip_matches_oracle,  # noqa: F401
                                  test_mip_rolled_view_reads_a_copy_bit_identically,
                                  test_sigma_clipping_matches_oracle, test_sigma_with_one_region_equals_rescaled_composite)
from tests.test_gpu_sortlast import (test_sub_cube_volumes_give_the_whole_volume_partials,  # noqa: F401
                                     test_subboxes_composite_to_the_whole_render)
from tests.test_gpu_sparse_groups import test_groups_match_single_lanes, test_small_dense_views  # noqa: F401
from tests.test_gpu_subbox_runs import test_runs_partition_every_ray  # noqa: F401
from tests.test_gpu_transparent import test_transparent_run_is_exact  # noqa: F401

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(autouse=True)
def ray_per_lane(monkeypatch):
    monkeypatch.setenv("VR_GROUPS", "0")


@pytest.mark.parametrize("layers", ["0", "1"])
def test_the_switch_picks_the_march(layers):
    cuda_or_skip()
    script = """
import os, torch, synth, paper_1211_4896_gb300 as P
vol = P.Volume(synth.hi_cube((40, 36, 44), 3, 0, 1).cuda(), "f32")
tf = torch.from_numpy(synth.tf_ramp(64)).cuda()
for g in ("0", "1", None):
    os.environ.pop("VR_GROUPS", None)
    if g: os.environ["VR_GROUPS"] = g
    for n in (8, 64, 256): P.render(vol, synth.camera_ortho((20, 18, -50), (0, 0, 1), (0, 1, 0), 36.0, n, n), tf, -3.0, 30.0, 0.5)
"""
    env = dict(os.environ, PYTHONPATH=ROOT, VR_LOG="1", VR_TEX_LAYERS=layers)
    r = subprocess.run([sys.executable, "-c", script], cwd=ROOT, env=env, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]
    lanes = [line.split(" lane(s)")[0].split()[-1] for line in r.stderr.splitlines() if " lane(s) to a ray" in line]
    assert lanes == ["1"] * 3 + ["8"] * 3 + ["8", "8", "1"]
