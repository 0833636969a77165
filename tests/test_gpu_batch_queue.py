"""Batches whose waits run out while more streams are tracked than are registered
at the same time: the streams whose registration did not finish report it, and
every volume registers normally afterwards, bit for bit as a fresh volume of
the same content does.  The waits run out by a limit of a few polls, or by one
arrival more than there are CTAs (fault injection through rf_set_wait_limits);
each ends by its limit."""
import numpy as np
import pytest

from synth.scenes import CAM_QVGA

from ._scenes import ROOM, look_at, render_frame
from .test_gpu_failures import BOX, NOT_CONVERGED, R, TARGET, _dev, _room_volume  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _volume(R, snap):  # noqa: F811
    vol = R.Volume(n_buckets=1 << 16, max_blocks=120000, max_width=CAM_QVGA.width, max_height=CAM_QVGA.height,
                   voxel_size=0.02, trunc=0.1)
    vol.import_(snap)
    return vol


@pytest.mark.parametrize("polls,extra", [(1, 0), (40, 0), (1 << 12, 1)])
def test_volumes_register_normally_after_a_batch_whose_waits_ran_out(R, polls, extra):  # noqa: F811
    n, cam = 6, CAM_QVGA
    room = _room_volume(R)
    snap = room.export()
    room.close()
    T = look_at([0.45, 0.32, 1.31], TARGET)
    d, rgb, _ = render_frame([ROOM, BOX], cam, T)
    vols = [_volume(R, snap) for _ in range(n)]
    cfg = vols[0].launch_config()
    cfg.batch_group = 2
    vols[0].set_launch_config(cfg)
    frames = [_dev(R, v, d, rgb, cam) for v in vols]
    T0 = torch.from_numpy(np.ascontiguousarray(T)).cuda()
    outs = [torch.zeros(4, 4, dtype=torch.float64, device="cuda") for _ in vols]
    for v, f in zip(vols, frames):
        v.process(f, T)
        v.sync()
        v.set_wait_limits(spin_limit=polls, extra_arrivals=extra)
    batch = R.Batch(vols)
    for _ in range(2):
        batch.process(frames, [T0] * n, outs)
        failed = 0
        for v in vols:
            try:
                v.sync()
            except R.RFError as e:
                assert e.status == NOT_CONVERGED and "grid-wide wait" in str(e)
                failed += 1
        if extra:  # (a limit of 40 polls may be enough)
            assert failed == n
        elif polls == 1:
            assert failed > 0
    batch.close()
    for v in vols:
        v.set_wait_limits(0, 0)
        fresh = _volume(R, v.export())
        for _ in range(2):
            got, _ = v.track(_dev(R, v, d, rgb, cam), T)
            want, _ = fresh.track(_dev(R, fresh, d, rgb, cam), T)
            v.sync()
            fresh.sync()
            np.testing.assert_array_equal(got.cpu().numpy(), want.cpu().numpy())
        fresh.close()
        v.close()
