"""Which of its two forms a run or a single image takes: the planes path (z
transformed first, its x-FFT a phase of its own) or the x-first passes.  The
choice is by cost; here are calls whose two sides differ by 1.25 times or
more, on the side that is the faster (x-first and planes, us, measured):
stacks whose z transform is a long direct sum, batches of one angle, one
angle alone."""
import pytest

from paper_2209_13121_gb300 import synth

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


# nx, ny, nz, voxel nm, precision, algorithm, angles (0: one image), planes?
CALLS = [(256, 256, 255, 2.0, 32, 1, 24, False),   # 11949, 44319
         (256, 256, 255, 2.0, 32, 1, 1, False),    # 505, 2614
         (256, 256, 255, 5.0, 32, 1, 0, False),    # 492, 1269
         (256, 256, 200, 2.0, 32, 1, 4, False),    # 1594, 2788
         (256, 256, 127, 2.0, 32, 2, 1, False),    # 287, 483
         (256, 2048, 9, 2.0, 32, 1, 24, False),    # 3831, 5720
         (128, 128, 255, 5.0, 64, 2, 4, False),    # 10125, 17923
         (128, 128, 191, 5.0, 64, 1, 0, False),    # 2252, 3728
         (1024, 512, 4, 5.0, 32, 1, 1, False),     # 90, 126
         (2048, 1024, 12, 2.2, 32, 1, 1, False),   # 665, 1119
         (512, 100, 127, 2.0, 32, 2, 1, False),    # 265, 402
         (32, 32, 4, 5.0, 32, 1, 0, False),        # 29, 38
         (32, 32, 4, 5.0, 32, 1, 8, True),         # 187, 48
         (256, 256, 64, 5.0, 32, 1, 0, True),      # 145, 112
         (256, 256, 64, 5.0, 32, 1, 24, True),     # 3307, 1375
         (300, 300, 16, 5.0, 32, 1, 4, True),      # 386, 164
         (97, 101, 255, 5.0, 32, 1, 1, True),      # 1170, 487
         (512, 512, 20, 5.0, 32, 1, 24, True),     # 3272, 1433
         (2048, 512, 16, 5.0, 32, 1, 8, True),     # 2956, 1333
         (128, 128, 64, 2.0, 64, 1, 0, True),      # ratio 1.4 and more
         (512, 512, 16, 5.0, 64, 2, 4, True),      # 7509, 3720
         (100, 100, 16, 5.0, 64, 1, 4, True)]


@pytest.mark.parametrize("nx,ny,nz,voxel,prec,alg,angles,planes", CALLS)
def test_the_faster_form_is_taken(rsx, nx, ny, nz, voxel, prec, alg, angles, planes):
    dt = torch.float32 if prec == 32 else torch.float64
    M = synth.morphology_random_torch((nz, ny, nx), 2, dtype=dt)
    K = synth.optical_constants([285.0], 2)
    out = torch.empty((1, ny, nx), device="cuda", dtype=dt)
    with rsx.Context(nx, ny, nz, 2, voxel, precision=prec, algorithm=alg) as ctx:
        ctx.set_morphology(M)
        ctx.set_optical_constants([285.0], K)
        ctx.set_timing(True)
        if angles:
            step = 180.0 / angles
            ctx.run((0.0, step, 180.0 - step), out=out)
        else:
            ctx.scatter_angle(0, 0.3, out[0])
        assert (ctx.phase_times()["fftx"][1] > 0) == planes
