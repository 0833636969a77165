"""The mask's erosion, flood fill and dilation on tiles of bits, at the sizes
where tiles, CTA regions and rows end, against the FP64 oracle bit for bit
(every step is integer arithmetic): corridors one pixel wide that wind through
the whole image (every tile border is crossed many times, in both
directions), and random depth steps around the threshold of Alg. 1 (its
conditions are directed)."""
import numpy as np
import pytest

from synth.scenes import Camera

from ._scenes import fronto_plane_frame

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

VOXEL, TAU, PLANE = 0.02, 0.1, 2000


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
    f = 1.3 * max(w, h)
    return Camera(w, h, f, f, (w - 1) / 2.0, (h - 1) / 2.0)


def _maze(w, h, pattern):
    """Depth in mm: corridors at 1.95 m between walls at 2.05 m (neither is a
    seed against the plane at 2 m: |V| = 5 cm), entered from a patch of seeds
    at 1.90 m over a ramp of steps below the threshold (0.7 %)."""
    d = np.full((h, w), PLANE + 50, np.uint16)
    if pattern == "random":
        rng = np.random.default_rng(w * 1000 + h)
        d[:] = PLANE - 50 + np.cumsum(rng.integers(-14, 15, (h, w)), axis=1) % 90
    elif pattern == "rows":
        for k, v in enumerate(range(1, h, 2)):
            d[v, :] = PLANE - 50
            if v + 1 < h:
                d[v + 1, -1 if k % 2 == 0 else 0] = PLANE - 50
    else:
        for k, u in enumerate(range(1, w, 2)):
            d[:, u] = PLANE - 50
            if u + 1 < w:
                d[-1 if k % 2 == 0 else 0, u + 1] = PLANE - 50
    v0, u0 = h // 3, w // 3  # the seeds, and a ramp around them
    for ring, mm in ((5, -50), (4, -60), (3, -70), (2, -80), (1, -90), (0, -100)):
        d[v0 - 3 - ring:v0 + 4 + ring, u0 - 3 - ring:u0 + 4 + ring] = PLANE + mm
    return d


def _model(O, cam):
    d, rgb = fronto_plane_frame(cam, PLANE)
    orc = O.OracleVolume(voxel_size=VOXEL, trunc=TAU)
    orc.integrate(O.FrameData(d, rgb, cam.fx, cam.fy, cam.cx, cam.cy), np.eye(4))
    snap = orc.export()
    snap["F"] = snap["F"].astype(np.float32).astype(np.float64)
    shared = O.OracleVolume(voxel_size=VOXEL, trunc=TAU)
    shared.import_(snap)
    return shared, snap


def _volume(R, cam, snap):
    vol = R.Volume(n_buckets=1 << 14, max_blocks=30000, max_width=cam.width, max_height=cam.height, voxel_size=VOXEL,
                   trunc=TAU)
    vol.import_(snap)
    return vol


def _device_frame(R, vol, d, rgb, cam):
    dt = torch.from_numpy(d.astype(np.int32)).cuda().to(torch.uint16).contiguous()
    ct = torch.from_numpy(np.ascontiguousarray(rgb)).cuda().contiguous()
    fr = vol.frame(dt, ct, R.Intrinsics(cam.fx, cam.fy, cam.cx, cam.cy))
    fr._keep = (dt, ct)
    return fr


@pytest.mark.parametrize("pattern", ["rows", "columns", "random"])
@pytest.mark.parametrize("size", [(31, 33), (32, 32), (33, 31), (65, 129), (130, 127), (257, 96), (320, 240)])
def test_mask_matches_oracle_at_tile_edges(R, oracle_mod, size, pattern):
    cam = _camera(*size)
    orc, snap = _model(oracle_mod, cam)
    d = _maze(*size, pattern)
    _, rgb = fronto_plane_frame(cam, PLANE)
    vol = _volume(R, cam, snap)
    got = vol.compute_mask(_device_frame(R, vol, d, rgb, cam), np.eye(4)).cpu().numpy()
    vol.sync()
    ref = orc.compute_mask(oracle_mod.FrameData(d, rgb, cam.fx, cam.fy, cam.cx, cam.cy), np.eye(4))
    assert ref.any()
    np.testing.assert_array_equal(got, ref)
    vol.close()


def test_batch_masks_with_fewer_ctas_than_regions(R, oracle_mod):
    """Sixteen 640x480 streams in one flood-fill launch get fewer CTAs each
    than the image has regions of 128 x 128 pixels, so a CTA works through
    several; the masks equal a single stream's."""
    n, cam = 16, _camera(640, 480)
    _, snap = _model(oracle_mod, cam)
    d = _maze(640, 480, "rows")
    d[200:280] = PLANE - 50  # (an open band: the maze's full corridor would take over a thousand sweeps)
    _, rgb = fronto_plane_frame(cam, PLANE)
    vols = [_volume(R, cam, snap) for _ in range(n + 1)]
    cfg = vols[0].launch_config()
    cfg.batch_group = 0
    vols[0].set_launch_config(cfg)
    frames = [_device_frame(R, v, d, rgb, cam) for v in vols]
    T0 = torch.eye(4, dtype=torch.float64, device="cuda")
    outs = [torch.empty(4, 4, dtype=torch.float64, device="cuda") for _ in vols]
    masks = [torch.empty(480, 640, dtype=torch.uint8, device="cuda") for _ in vols]
    batch = R.Batch(vols[:n])
    batch.process(frames[:n], [T0] * n, outs[:n], masks[:n])
    R.rf_process_frame(vols[n].h, frames[n], T0, outs[n], masks[n], None)
    for v in vols:
        v.sync()
    assert int(masks[n].sum()) > 1000
    for k in range(n):
        np.testing.assert_array_equal(masks[k].cpu().numpy(), masks[n].cpu().numpy())
    batch.close()
    for v in vols:
        v.close()


def test_batch_masks_with_far_fewer_ctas_than_regions(R, oracle_mod):
    """Enough 640x480 streams in one flood-fill launch that each has fewer CTAs
    than regions whatever the kernel's occupancy (512 threads: at most 4 CTAs
    per SM); the masks equal the oracle's at the streams' own poses."""
    cam, regions = _camera(640, 480), 5 * 4
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = 4 * sms // regions + 1
    assert n <= sms and 4 * sms // n < regions
    orc, snap = _model(oracle_mod, cam)
    _, rgb = fronto_plane_frame(cam, PLANE)
    depths = [_maze(640, 480, p) for p in ("rows", "columns", "random")]
    depths[0][200:280] = PLANE - 50  # (open bands: the full corridors would take over a thousand sweeps)
    depths[1][:, 280:360] = PLANE - 50
    vols = [_volume(R, cam, snap) for _ in range(n)]
    cfg = vols[0].launch_config()
    cfg.batch_group = 0
    vols[0].set_launch_config(cfg)
    frames = [_device_frame(R, v, depths[k % 3], rgb, cam) for k, v in enumerate(vols)]
    T0 = torch.eye(4, dtype=torch.float64, device="cuda")
    # the pose of a stream's mask: its first registration, as the batch's bit for bit
    poses = [vols[k].track(frames[k], T0)[0].cpu().numpy() for k in range(3)]
    outs = [torch.empty(4, 4, dtype=torch.float64, device="cuda") for _ in vols]
    masks = [torch.empty(480, 640, dtype=torch.uint8, device="cuda") for _ in vols]
    batch = R.Batch(vols)
    batch.process(frames, [T0] * n, outs, masks)
    for v in vols:
        v.sync()
    want = [orc.compute_mask(oracle_mod.FrameData(d, rgb, cam.fx, cam.fy, cam.cx, cam.cy), T)
            for d, T in zip(depths, poses)]
    assert all(w.any() for w in want) and max(int(w.sum()) for w in want) > 1000
    for k in range(n):
        np.testing.assert_array_equal(masks[k].cpu().numpy(), want[k % 3])
    batch.close()
    for v in vols:
        v.close()
