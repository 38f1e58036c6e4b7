"""Device memory of a context (host arithmetic, no GPU): angle_batch = 1 asks for
the least on every shape, and the default's extra is bounded."""
import pytest

from paper_2209_13121_gb300 import rsx

MB = 1 << 20

# nx, ny, nz, c, precision, algorithm
SHAPES = [(256, 256, 32, 4, 64, 1), (256, 256, 32, 4, 64, 2), (300, 180, 45, 3, 32, 1),
          (128, 128, 16, 4, 32, 1), (100, 100, 255, 2, 32, 2), (256, 256, 64, 6, 32, 2),
          (512, 512, 1, 2, 32, 1), (1000, 1000, 1, 2, 64, 1), (1024, 1024, 32, 4, 32, 2),
          (24, 40, 7, 3, 64, 1)]


def _least(nx, ny, nz, c, prec, alg):
    """Tables 1 and 2: the morphology copy or N_t and its staging, one p, two
    images; and per pixel the Ewald geometry (32 or 64 bytes), a bin index and
    the partial bins of the fused y and z pass (FP32), per slice 16 numbers,
    twiddles; FP64 Algorithm 1 the director of every voxel."""
    r, n, npix = prec // 8, nx * ny * nz, nx * ny
    b = 4 * c * n * r if alg == 1 else 10 * n * r + 8 * min(n, 1 << 22) * r
    b += 6 * n * r + 2 * npix * r + npix * (32 if prec == 32 else 64)
    if prec == 64 and alg == 1:
        b += 3 * c * n * r
    if prec == 32:
        b += (2 + 192) * npix
    return b + 16 * nz * r + 2 * r * (nx + ny + nz) + 64


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_angle_batch_one_holds_one_p_and_one_image(shape):
    nx, ny, nz, c, prec, alg = shape
    got = rsx.workspace_bytes(rsx.make_config(nx, ny, nz, c, 5.0, precision=prec, algorithm=alg,
                                              angle_batch=1))
    assert 0 < got <= _least(*shape)


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_the_defaults_extra_is_bounded(shape):
    nx, ny, nz, c, prec, alg = shape

    def at(k):
        return rsx.workspace_bytes(rsx.make_config(nx, ny, nz, c, 5.0, precision=prec,
                                                   algorithm=alg, angle_batch=k))
    p = 3 * nx * ny * nz * prec // 4
    pool = (96 if prec == 32 else 1024) * MB
    tuned = 7 * p if prec == 32 and alg == 1 and nx in (512, 1024, 2048) else 0
    assert at(1) <= at(2) <= at(8) <= at(0) <= at(1) + max(tuned, min(31 * p, pool)) + 64 * MB
