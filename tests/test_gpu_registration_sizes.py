"""Registration against the FP64 oracle at frame sizes where its chunks, slots
and levels end: fewer samples than one chunk of 128, a level of one chunk and a
few pixels, chunks that are not a whole number of CTA widths, odd rows.  The
bar is the repository's: 1e-4 m and 1e-4 rad; scenes without noise, so that
every level converges."""
import numpy as np
import pytest

from synth.scenes import Camera

from ._scenes import ROOM, SPHERE, corner_pose, render_frame, rot_err

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SIZES = [(26, 19), (43, 31), (97, 73), (161, 121), (259, 197), (403, 301)]


@pytest.fixture(scope="module")
def R():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1905_02082_gb300 import build as B
    B.build()
    import paper_1905_02082_gb300.refusion as R
    R.load()
    return R


def _camera(w, h):
    f = 130.0 * w / 160.0
    return Camera(w, h, f, f, (w - 1) / 2.0, (h - 1) / 2.0)


@pytest.mark.parametrize("masked", [False, True])
@pytest.mark.parametrize("size", SIZES)
def test_registration_matches_oracle(R, oracle_mod, size, masked):
    O, cam = oracle_mod, _camera(*size)
    src = O.OracleVolume(voxel_size=0.02, trunc=0.1)
    for i in range(3):
        T = corner_pose(i)
        d, rgb, _ = render_frame([ROOM, SPHERE], _camera(259, 197), T)
        c = _camera(259, 197)
        src.integrate(O.FrameData(d, rgb, c.fx, c.fy, c.cx, c.cy), T)
    snap = src.export()
    snap["F"] = snap["F"].astype(np.float32).astype(np.float64)
    orc = O.OracleVolume(voxel_size=0.02, trunc=0.1)
    orc.import_(snap)
    vol = R.Volume(n_buckets=1 << 14, max_blocks=40000, max_width=cam.width, max_height=cam.height, voxel_size=0.02,
                   trunc=0.1)
    vol.import_(snap)
    T = corner_pose(1.5)
    d, rgb, _ = render_frame([ROOM, SPHERE], cam, T)
    mask = None
    if masked:
        mask = np.zeros(d.shape, np.uint8)
        mask[: cam.height // 3, : cam.width // 2] = 1
    T0 = corner_pose(1.0)
    dt = torch.from_numpy(d.astype(np.int32)).cuda().to(torch.uint16).contiguous()
    ct = torch.from_numpy(np.ascontiguousarray(rgb)).cuda().contiguous()
    fr = vol.frame(dt, ct, R.Intrinsics(cam.fx, cam.fy, cam.cx, cam.cy))
    got, info = vol.track(fr, T0, mask=None if mask is None else torch.from_numpy(mask).cuda())
    vol.sync()
    got = got.cpu().numpy()
    ref, oinfo = orc.track(O.FrameData(d, rgb, cam.fx, cam.fy, cam.cx, cam.cy), T0, mask)
    assert np.linalg.norm(got[:3, 3] - ref[:3, 3]) < 1e-4
    assert rot_err(got[:3, :3], ref[:3, :3]) < 1e-4
    gi = R.Volume.info_of(info)
    assert abs(gi.final_valid - oinfo.final_valid) <= 0.01 * oinfo.final_valid
    vol.close()
