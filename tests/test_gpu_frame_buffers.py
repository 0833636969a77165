"""rf_process_frame from and to the buffers it accepts: a frame in device,
page-locked or pageable memory (the last by copies), its pose and results in
device or page-locked memory.  Every kind gives the same pose, mask and info,
byte for byte."""
import numpy as np
import pytest

from synth.scenes import CAM_QVGA

from ._scenes import ROOM, look_at, render_frame
from .test_gpu_failures import BOX, R, TARGET, _room_volume  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _run(R, snap, place):  # noqa: F811
    cam = CAM_QVGA
    room = R.Volume(n_buckets=1 << 16, max_blocks=120000, max_width=cam.width, max_height=cam.height, voxel_size=0.02,
                    trunc=0.1)
    room.import_(snap)
    got = []
    for k in range(2):
        T = look_at([0.45 + 0.01 * k, 0.32, 1.31], TARGET)
        d, rgb, _ = render_frame([ROOM, BOX], cam, T)
        depth, colour = place(torch.from_numpy(d.view(np.int16).copy())), place(torch.from_numpy(rgb.copy()))
        results = place if place is not _pageable else _device
        pose = results(torch.from_numpy(np.ascontiguousarray(T)))
        out, mask = results(torch.zeros(4, 4, dtype=torch.float64)), results(torch.zeros(cam.height, cam.width,
                                                                                        dtype=torch.uint8))
        info = results(torch.zeros(R.C.sizeof(R.rf_track_info), dtype=torch.uint8))
        frame = R.rf_frame(cam.height, cam.width, cam.fx, cam.fy, cam.cx, cam.cy, depth.data_ptr(), colour.data_ptr())
        R.rf_process_frame(room.h, frame, pose, out, mask, info, None)
        room.sync()
        got += [t.cpu().numpy().copy() for t in (out, mask, info)]
    room.close()
    return got


def _device(t):
    return t.cuda()


def _pinned(t):
    return t.pin_memory()


def _pageable(t):
    return t


@pytest.mark.parametrize("place", [_pinned, _pageable])
def test_frame_and_results_in_other_memory(R, place):  # noqa: F811
    room = _room_volume(R)
    snap = room.export()
    room.close()
    for a, b in zip(_run(R, snap, _device), _run(R, snap, place)):
        assert a.any()
        np.testing.assert_array_equal(a, b)
