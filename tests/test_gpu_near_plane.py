"""A surface that lies on the near plane: its vertices fall on one side or the
other by FP32 rounding alone, and the oracle clips the triangles that have one in
front.  The set-up drops a cluster of cells by the corners of the frustum piece that
holds it, which are other points with other roundings, so it may do so only with a
margin for them.

The scene: a camera some kilometres to the eye's left whose first column of rays is
perpendicular to the eye's axis, so that this column's vertices have the eye depth
z_near whatever their distance, up to a few rounding errors of that distance; every
other column lies behind.  Per case the yaw, the distance, each row's distance in ulps
beyond it, and the camera's offset from the eye: values for which the nearest and the
farthest vertex round to a depth below z_near and two rows between them do not."""
import math

import numpy as np
import pytest

import oracle
import scene
from tests import lfcase
from tests.test_gpu_parity import _check_full_frame

pytestmark = pytest.mark.gpu

CASES = [
    (0.8666156139816421, -169.8920872740592, 10826.9755859375, (3, 9, 8, 11, 2), -14205.970966207842, 0.10040673424170989),
    (0.8775952023829459, -166.1463929417033, 7583.93896484375, (8, 2, 3, 7, 2), -9859.473915110952, 0.09952718737676854),
    (0.8991632132288506, -158.98315963608377, 8137.45166015625, (0, 7, 4, 6, 5), -10395.225284022024, 0.09994576243384086),
    (0.9074566190097078, -156.2940294057028, 198681.140625, (4, 10, 3, 1, 4), -252152.61862949913, 0.09241164432922253),
]


def _field(grid, yaw, cx, z, ulps, mx, mz):
    """The light field of one view: columns 0.01 apart in slope from -cx / 200 on, rows 0.005 apart."""
    size = 2 * (grid - 1)
    c, s = math.cos(yaw), math.sin(yaw)
    pose = [c, 0, s, 0, 1, 0, -s, 0, c, mx, 0, mz]
    z = np.float32(z)
    rows = np.array([z + np.float32(np.spacing(z) * u) for u in ulps + (min(ulps),) * (grid - 5)], np.float32)
    return lfcase.custom_lf([pose], [[200.0, 400.0, cx, 4.0]], np.full((1, size, size, 4), 200, np.uint8),
                            np.repeat(rows[:, None], grid, 1)[None], disk_c=[[0, 0, 0.3]], disk_r=[2.0])


@pytest.mark.parametrize("case", CASES)
@pytest.mark.parametrize("grid", [5, 69])  # one cluster; a set-up of several blocks per view
def test_clusters_on_the_near_plane_are_clipped_as_the_oracle_clips_them(grid, case):
    pytest.importorskip("torch")
    import __graft_entry__

    __graft_entry__.build()
    import paper_1810_08860_gb300 as lfm

    lf = _field(grid, *case)
    eye = scene.Eye(scene.pose_array(np.eye(3), (0, 0, 0)), np.array([100.0, 100.0, 20.0, 16.0]), 40, 32)
    assert (oracle.render(lf, eye)["rgba"][..., 3] > 0).any()
    r = lfm.Renderer(0)
    r.load_views(lf)
    r.build_meshes(lf)
    _check_full_frame(r, lf, eye)
    r.close()
