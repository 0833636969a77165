"""Virtual depth visits only the samples inside the bounds of the allocated
blocks: from cameras inside and outside those bounds, along the axes (ray
directions with zero components) and across them, and from a camera that sees
none of them, every filled depth equals the FP64 oracle's, bit for bit."""
import numpy as np
import pytest

from synth.scenes import Camera

from ._scenes import look_at

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CAM = Camera(41, 33, 40.0, 40.0, 20.0, 16.0)  # pixel (20, 16) looks exactly along the axis
VOXEL, TAU = 0.02, 0.1


@pytest.fixture(scope="module")
def R():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1905_02082_gb300 import build as B
    B.build()
    import paper_1905_02082_gb300.refusion as R
    R.load()
    return R


def _axis_pose(z):
    T = np.eye(4)
    T[2, 3] = z
    return T


POSES = {"inside": _axis_pose(0.0), "behind": _axis_pose(-1.5), "turned": look_at([0.9, -0.4, -0.8], np.array([0.1, 0.1, 1.4])),
         "away": look_at([0.0, 0.0, 3.0], np.array([0.2, 0.1, 4.0])), "far off": look_at([5.0, 0.0, 0.0], np.array([5.0, 0.3, 2.0]))}


@pytest.mark.parametrize("storage", ["fp32", "fp16"])
@pytest.mark.parametrize("pose", list(POSES))
def test_rays_clipped_to_the_model_match_the_oracle(R, oracle_mod, pose, storage):
    O = oracle_mod
    v, u = np.mgrid[0:CAM.height, 0:CAM.width]
    d = (1200 + 6 * u + 3 * v).astype(np.uint16)  # a slanted surface
    rgb = np.full((CAM.height, CAM.width, 3), 90, np.uint8)
    src = O.OracleVolume(voxel_size=VOXEL, trunc=TAU)
    src.integrate(O.FrameData(d, rgb, CAM.fx, CAM.fy, CAM.cx, CAM.cy), np.eye(4))
    snap = src.export()
    F = snap["F"].astype(np.float32)
    if storage == "fp16":
        F = (F / np.float32(TAU)).astype(np.float16).astype(np.float32) * np.float32(TAU)
    snap["F"] = F.astype(np.float64)
    orc = O.OracleVolume(voxel_size=VOXEL, trunc=TAU)
    orc.import_(snap)
    vol = R.Volume(n_buckets=1 << 13, max_blocks=20000, max_width=CAM.width, max_height=CAM.height, voxel_size=VOXEL,
                   trunc=TAU, storage=R.STORAGE_FP16 if storage == "fp16" else R.STORAGE_FP32)
    vol.import_(snap)
    hole = np.zeros_like(d)
    hole[::7, ::5] = 777  # a few pixels with depth, copied
    dt = torch.from_numpy(hole.astype(np.int32)).cuda().to(torch.uint16).contiguous()
    ct = torch.from_numpy(rgb).cuda()
    fr = vol.frame(dt, ct, R.Intrinsics(CAM.fx, CAM.fy, CAM.cx, CAM.cy))
    T = POSES[pose]
    got = vol.virtual_depth(fr, T).to(torch.int32).cpu().numpy()
    vol.sync()
    ref = np.asarray(orc.virtual_depth(O.FrameData(hole, rgb, CAM.fx, CAM.fy, CAM.cx, CAM.cy), T)).astype(np.int32)
    np.testing.assert_array_equal(got, ref)
    if pose in ("inside", "behind", "turned"):
        assert (got[hole == 0] < 5000).any()
    vol.close()
