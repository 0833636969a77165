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
        got += [t.cpu().numpy().copy() for t in (out, mask)]
        i = R.rf_track_info.from_buffer_copy(info.cpu().numpy().tobytes())  # (field by field: it has padding)
        got.append(np.hstack([np.ravel(np.ctypeslib.as_array(x) if hasattr(x, "__len__") else x).astype(np.float64)
                              for x in (getattr(i, name) for name, _ in i._fields_)]))
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


def _offset(nbytes, pin=False):
    def place(t):
        raw = t.contiguous().view(torch.uint8).reshape(-1)
        room = torch.zeros(raw.numel() + 16, dtype=torch.uint8)
        room = room.pin_memory() if pin else room.cuda()
        room[nbytes:nbytes + raw.numel()] = raw
        return room[nbytes:nbytes + raw.numel()]
    return place


@pytest.mark.parametrize("nbytes,pin", [(2, False), (4, False), (8, False), (2, True)])
def test_unaligned_frame_and_results(R, nbytes, pin):  # noqa: F811
    """Views into larger buffers, as the frames of a stack whose frame size is
    not a multiple of 16 bytes, at offsets that the images' element size allows."""
    room = _room_volume(R)
    snap = room.export()
    room.close()
    for a, b in zip(_run(R, snap, _device), _run(R, snap, _offset(nbytes, pin))):
        np.testing.assert_array_equal(a.reshape(-1).view(np.uint8), b.reshape(-1).view(np.uint8))
