"""More of the planes path against the oracle: the pass of 1024-voxel tiles on
lateral sizes of no tuned kernel and with more than half the bins kept (its
whole-transform form), each tuned y pass behind the general p + z pass, a
fresh context after a timeout, and the smallest workspace."""
import math

import numpy as np
import pytest

from oracle import cyrsoxs_oracle as O
from paper_2209_13121_gb300 import synth
from tests.test_gpu_planes import _close

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def rsx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2209_13121_gb300 import rsx as R
    return R


def _kept(nx, ny, nz, voxel, E):
    """Bins the pixels read, to within one."""
    k = 2 * math.pi * E / 1239.84198
    q = 2 * math.pi * np.hypot(np.fft.fftfreq(nx, voxel)[None], np.fft.fftfreq(ny, voxel)[:, None])
    q = q[q <= k].max()
    return 2 + math.ceil((k - math.sqrt(k * k - q * q)) * nz * voxel / (2 * math.pi))


# (nz, ny, nx), voxel nm, energy eV, more than half the bins kept
TILES = [((32, 103, 96), 5.0, 285.0, False), ((32, 103, 96), 2.8, 300.0, True),
         ((64, 75, 80), 5.0, 285.0, False), ((64, 75, 80), 2.8, 300.0, True),
         ((128, 51, 56), 5.0, 285.0, False), ((128, 51, 56), 2.8, 300.0, True)]


@pytest.mark.parametrize("frame", [0, 1])
@pytest.mark.parametrize("shape,voxel,E,whole", TILES,
                         ids=["x".join(map(str, t[0])) + f"@{t[1]:g}nm" for t in TILES])
def test_tile_pass_on_general_lateral_sizes(rsx, shape, voxel, E, whole, frame):
    nz, ny, nx = shape
    # the pass is taken from two tiles per SM on, rows in whole tiles
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert nx * ny * nz >= 2048 * sms and nx % (1024 // nz) == 0
    kept = _kept(nx, ny, nz, voxel, E)
    assert kept > nz // 2 + 1 if whole else kept <= nz // 2
    c, angles = 3, (0.0, 30.0, 150.0)
    M = synth.morphology_random(shape, c, seed=31, dtype=np.float32)
    K = synth.optical_constants([E], c, seed=32)
    ref = O.run_alg1(M, K, [E], voxel, angles_deg=angles, uT_mode="lab" if frame else "literal")
    with rsx.Context(nx, ny, nz, c, voxel, frame=frame) as ctx:
        ctx.set_morphology(torch.from_numpy(M).cuda())
        ctx.set_optical_constants([E], K)
        ctx.set_timing(True)
        got = ctx.run(angles)
        assert ctx.phase_times()["fftx"][1] > 0  # the planes path
        _close(got, ref, 32)
        img = torch.empty((ny, nx), device="cuda")
        ctx.scatter_angle(0, 0.7, img)
    one = O.scatter_one_angle(M, K[0], E, voxel, 0.7, uT_mode="lab" if frame else "literal")
    _close(img.cpu().numpy(), one, 32, r=1.5)


@pytest.mark.parametrize("shape", [(16, 512, 32), (16, 1024, 32), (16, 2048, 16)],
                         ids=["512", "1024", "2048"])
def test_y_pass_matches_the_oracle_and_recovers_to_a_fresh_contexts_result(rsx, shape):
    """The tuned y passes behind the general p + z pass, against the oracle; and
    a context whose waits ran out gives, with the default bound restored, the
    result of another context that never failed, bit for bit."""
    nz, ny, nx = shape
    angles = (0.0, 30.0, 150.0)
    M = synth.morphology_random(shape, 2, seed=15, dtype=np.float32)
    K = synth.optical_constants([285.0], 2, seed=16)
    dev = torch.from_numpy(M).cuda()
    with rsx.Context(nx, ny, nz, 2, 5.0) as fresh:
        fresh.set_morphology(dev)
        fresh.set_optical_constants([285.0], K)
        want = fresh.run(angles)
    _close(want, O.run_alg1(M, K, [285.0], 5.0, angles_deg=angles), 32)
    with rsx.Context(nx, ny, nz, 2, 5.0) as ctx:
        ctx.set_morphology(dev)
        ctx.set_optical_constants([285.0], K)
        ctx.set_wait_limit(0)
        with pytest.raises(rsx.RsxError):
            ctx.run(angles)
        ctx.set_wait_limit()
        np.testing.assert_array_equal(ctx.run(angles), want)


@pytest.mark.parametrize("shape,prec,alg", [((16, 20, 52), 32, 1), ((45, 12, 11), 64, 1),
                                            ((16, 20, 52), 64, 2), ((30, 33, 17), 32, 2),
                                            ((1, 24, 40), 32, 1), ((16, 64, 512), 32, 1)])
def test_smallest_workspace_gives_the_same_images(rsx, shape, prec, alg):
    """angle_batch = 1 (one p, one image) and 3 against the default: the same
    arithmetic per angle in other batches, or the other form of the path, so
    the parity tolerances hold between them."""
    nz, ny, nx = shape
    M = synth.morphology_random(shape, 2, seed=33, dtype=np.float32 if prec == 32 else np.float64)
    K = synth.optical_constants([285.0], 2, seed=34)
    out = {}
    for k in (0, 1, 3):
        with rsx.Context(nx, ny, nz, 2, 5.0, precision=prec, algorithm=alg, angle_batch=k) as ctx:
            ctx.set_morphology(torch.from_numpy(M).cuda())
            ctx.set_optical_constants([285.0], K)
            out[k] = ctx.run((0.0, 15.0, 165.0))
    _close(out[1], out[0], prec)
    _close(out[3], out[0], prec)
