"""The general planes path of rsx_run (Algorithms 1 and 2, nz <= 255, both
precisions): per pixel column p and its z transform at only the q_z bins the
detector reads, the lateral transforms of those planes, images and rotation
for a batch of angles at a time.  Checked at the edges of its rules: one
slice, odd and even stacks, the tallest stack it takes and the first beyond
it, pixel tiles with a remainder, runs of bins that wrap onto themselves,
energies and voxels that read few or nearly all bins, more angles than a
batch holds."""
import numpy as np
import pytest

from oracle import cyrsoxs_oracle as O
from paper_2209_13121_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

# the parity tests' tolerances: relative L2 away from q = 0, per pixel above a floor
TOL = {64: dict(norm=1e-10, pix=1e-8, floor=1e-8), 32: dict(norm=1e-4, pix=2e-3, floor=1e-4)}


@pytest.fixture(scope="module")
def rsx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2209_13121_gb300 import rsx as R
    return R


def _close(got, ref, prec, r=2.5):
    got, ref = np.asarray(got, np.float64), np.asarray(ref, np.float64)
    ny, nx = ref.shape[-2:]
    iy, ix = np.meshgrid(np.arange(ny) - ny // 2, np.arange(nx) - nx // 2, indexing="ij")
    far = np.broadcast_to(np.hypot(ix, iy) > r, ref.shape)
    t = TOL[prec]
    assert np.all(np.isfinite(got))
    if far.any() and np.abs(ref[far]).max() > 0:
        assert np.linalg.norm((got - ref)[far]) <= t["norm"] * np.linalg.norm(ref[far])
    big = np.abs(ref) > t["floor"] * np.abs(ref).max()
    assert (np.abs(got - ref)[big] / np.abs(ref)[big]).max() <= t["pix"]


# (nz, ny, nx), c, voxel nm, energy eV
EDGES = [((1, 24, 40), 2, 5.0, 285.0), ((2, 9, 10), 3, 5.0, 285.0), ((3, 16, 64), 2, 5.0, 270.0),
         ((16, 20, 52), 3, 5.0, 285.0), ((45, 12, 11), 2, 5.0, 285.0), ((64, 8, 24), 2, 2.0, 300.0),
         ((127, 6, 10), 2, 5.0, 285.0), ((128, 8, 8), 2, 5.0, 285.0), ((254, 4, 6), 1, 5.0, 285.0),
         ((255, 3, 7), 2, 5.0, 285.0), ((256, 4, 4), 1, 5.0, 285.0), ((16, 16, 16), 2, 5.0, 60.0),
         ((32, 10, 12), 2, 1.0, 17000.0), ((30, 33, 17), 4, 10.0, 310.0)]


@pytest.mark.parametrize("prec", [32, 64])
@pytest.mark.parametrize("shape,c,voxel,E", EDGES,
                         ids=["x".join(map(str, e[0])) + f"@{e[3]:g}" for e in EDGES])
def test_edges_match_oracle_and_the_general_path(rsx, shape, c, voxel, E, prec):
    nz, ny, nx = shape
    M = synth.morphology_random(shape, c, seed=11, dtype=np.float32 if prec == 32 else np.float64)
    K = synth.optical_constants([E], c, seed=12)
    dev = torch.from_numpy(M).cuda()
    for alg, frame in ((1, 0), (2, 1)):
        ref = O.run_alg1(M, K, [E], voxel, angles_deg=(0.0, 40.0, 160.0),
                         uT_mode="lab" if frame else "literal")
        with rsx.Context(nx, ny, nz, c, voxel, precision=prec, algorithm=alg, frame=frame) as ctx:
            ctx.set_morphology(dev)
            ctx.set_optical_constants([E], K)
            _close(ctx.run((0.0, 40.0, 160.0)), ref, prec)
            # one angle without rotation is the single image, which keeps the
            # one-angle passes on small powers of two and FP32 rows of 512 and
            # 1024 points, and takes the planes path elsewhere
            img = torch.empty((ny, nx), device="cuda", dtype=dev.dtype)
            ctx.scatter_angle(0, 0.0, img)
            _close(ctx.run(rotation=False)[0], img.cpu().numpy(), prec, r=1.5)


# stacks the linearity path's z-first pass takes and their neighbours, the
# tuned x and y passes, both sources of N_t
LIN = [((7, 9, 10), 64), ((8, 12, 20), 32), ((16, 16, 32), 64), ((32, 10, 9), 32), ((64, 8, 8), 64),
       ((64, 8, 12), 32), ((128, 6, 10), 32), ((128, 4, 6), 64), ((16, 512, 16), 32),
       ((16, 1024, 16), 32), ((16, 4, 1024), 32), ((16, 3, 2048), 32)]


@pytest.mark.parametrize("shape,prec", LIN, ids=["x".join(map(str, s)) + f"f{p}" for s, p in LIN])
def test_linearity_path_planes(rsx, shape, prec):
    nz, ny, nx = shape
    E = [285.0, 300.0]
    M = synth.morphology_random(shape, 2, seed=17, dtype=np.float32 if prec == 32 else np.float64)
    K = synth.optical_constants(E, 2, seed=18)
    for dev, frame in ((True, 0), (False, 1)):
        ref = O.run_alg1(M, K, E, 5.0, angles_deg=(0.0, 40.0, 160.0),
                         uT_mode="lab" if frame else "literal")
        with rsx.Context(nx, ny, nz, 2, 5.0, precision=prec, algorithm=3, frame=frame) as ctx:
            ctx.set_morphology(torch.from_numpy(M).cuda() if dev else M)
            ctx.set_optical_constants(E, K)
            _close(ctx.run((0.0, 40.0, 160.0)), ref, prec)


FILMS = [(512, 512), (512, 1024), (1024, 512), (2048, 512), (512, 2048), (512, 2000)]


@pytest.mark.parametrize("ny,nx", FILMS, ids=[f"{a}x{b}" for a, b in FILMS])
def test_films_match_oracle(rsx, ny, nx):
    """One slice: p x-transformed by the multi-angle pass straight into the
    planes (rows of 512, 1024, 2048 points), each tuned column length, the
    2048-row columns' own kernel, a partial batch of angles; and a row length
    the multi-angle pass does not take."""
    M = synth.morphology_random((1, ny, nx), 2, seed=19, dtype=np.float32)
    K = synth.optical_constants([285.0], 2, seed=20)
    ref = O.run_alg1(M, K, [285.0], 5.0, angles_deg=(0.0, 45.0, 180.0))
    with rsx.Context(nx, ny, 1, 2, 5.0) as ctx:
        ctx.set_morphology(torch.from_numpy(M).cuda())
        ctx.set_optical_constants([285.0], K)
        _close(ctx.run((0.0, 45.0, 180.0)), ref, 32)


def test_more_angles_than_one_batch_holds(rsx):
    """181 angles in three or more batches of at most 64; two energies."""
    shape, c, E = (6, 12, 20), 2, [275.0, 300.0]
    M = synth.morphology_random(shape, c, seed=13, dtype=np.float32)
    K = synth.optical_constants(E, c, seed=14)
    ref = O.run_alg1(M, K, E, 5.0, angles_deg=(0.0, 1.0, 180.0))
    with rsx.Context(20, 12, 6, c, 5.0) as ctx:
        ctx.set_morphology(M)
        ctx.set_optical_constants(E, K)
        _close(ctx.run((0.0, 1.0, 180.0)), ref, 32)


@pytest.mark.parametrize("shape", [(16, 512, 32), (16, 1024, 32), (16, 2048, 16)],
                         ids=["512", "1024", "2048"])
def test_y_pass_timeout_is_reported_and_recoverable(rsx, shape):
    """With a wait bound of zero polls the y pass of the planes gives up
    cleanly: the run reports it, leaves its host output alone, and with the
    default bound restored gives a fresh context's result bit for bit."""
    nz, ny, nx = shape
    M = torch.from_numpy(synth.morphology_random(shape, 2, seed=15, dtype=np.float32)).cuda()
    K = synth.optical_constants([285.0], 2, seed=16)
    with rsx.Context(nx, ny, nz, 2, 5.0) as ctx:
        ctx.set_morphology(M)
        ctx.set_optical_constants([285.0], K)
        ref = ctx.run((0.0, 30.0, 150.0))
        out = np.full((1, ny, nx), 7.0, dtype=np.float32)
        ctx.set_wait_limit(0)
        with pytest.raises(rsx.RsxError) as e:
            ctx.run((0.0, 30.0, 150.0), out=out)
        assert e.value.code == rsx.RSX_ERR_CUDA and np.all(out == 7.0)
        ctx.set_wait_limit()
        np.testing.assert_array_equal(ctx.run((0.0, 30.0, 150.0)), ref)
