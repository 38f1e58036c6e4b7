"""FP32 accuracy where a kernel could drop bits without leaving the wide parity
tolerances: each bound here follows from the arithmetic the kernel is meant
to do, and is stated at the test."""
import math

import numpy as np
import pytest

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


@pytest.mark.parametrize("prec", [32, 64])
@pytest.mark.parametrize("bits", [12, 28, 36])
def test_rotation_weights_keep_all_fraction_bits(rsx, bits, prec):
    """Rotation by alpha = 2^-bits of an image with one nonzero column, the one
    beside the centre: the centre column gets the weight |dy| sin(alpha).  The
    source position is in 2^-48 fixed point, so its fraction is off by at most
    |dy| 2^-49 (a relative 2^(bits-49); for 28 and 36 the coefficients are
    whole multiples of 2^-48 and it is exact); the weight, 1 - ty, their
    product and the sum over the two rows are rounded once each: 5 units
    (2^-24 or 2^-53) bound them."""
    n = 64
    alpha = 2.0 ** -bits
    img = torch.zeros((n, n), device="cuda", dtype=torch.float32 if prec == 32 else torch.float64)
    img[:, n // 2 + 1] = 1.0
    acc = torch.zeros_like(img)
    with rsx.Context(n, n, 1, 1, 5.0, precision=prec) as ctx:
        ctx.rotate_accumulate(img, alpha, acc)
    got = acc.double().cpu().numpy()[:, n // 2]
    dy = np.arange(n) - n // 2
    want = np.where(dy < 0, -dy * math.sin(alpha), 0.0)
    inside = (dy < -1) & (dy > -n // 2)
    tol = 5 * 2.0 ** -24 if prec == 32 else 5 * 2.0 ** -53 + 2.0 ** (bits - 49)
    assert np.all(np.abs(got - want)[inside] <= tol * want[inside]), (got, want)


# (nz, ny, nx): register-FFT stacks, folded ones (even, odd), the pass of 1024-voxel tiles
FAINT = [(16, 24, 20), (45, 20, 24), (62, 20, 18), (64, 20, 24), (128, 12, 20), (32, 101, 96),
         (64, 75, 80)]


# Algorithm 3 transforms z first for the register-FFT stacks alone
@pytest.mark.parametrize("shape,alg", [(sh, a) for sh in FAINT for a in (1, 2, 3)
                                       if a < 3 or sh[0] & (sh[0] - 1) == 0],
                         ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else f"alg{v}")
def test_a_uniform_background_leaves_no_rounding_in_faint_images(rsx, shape, alg):
    """One unaligned material with v = 0.5 + 0.01 x, x uniform and white: the
    contrast v^2 - 1 has a mean near -0.75 and a standard deviation s of about
    0.003 per voxel.  Forming it and dividing it by 4 pi rounds twice at that
    size (at most 2^-25 each, root mean square 2^-25 sqrt(2/3) together), and
    a white error below a white signal is the image's relative L2 error away
    from q = 0; the transforms of a field without its mean add far less.  A
    mean that is still there when z is transformed adds nz roundings of its
    size to bin 0 and grows the error as sqrt(nz).  Bound: 2 2^-25 / s.  Eight
    angles of 0 and 180 degrees, whose rotations are exact, so that the planes
    path is taken."""
    from oracle import cyrsoxs_oracle as O
    from paper_2209_13121_gb300 import synth
    nz, ny, nx = shape
    M = np.zeros((1, nz, ny, nx, 4), dtype=np.float32)
    M[..., 0] = 0.5 + 0.01 * np.random.default_rng(5).random((nz, ny, nx))
    K = synth.optical_constants([285.0], 1, seed=6)
    s = float(np.std(M[..., 0].astype(np.float64) ** 2))
    angles = (0.0, 180.0, 1260.0)
    ref = O.run_alg1(M.astype(np.float64), K, [285.0], 5.0, angles_deg=angles)[0]
    iy, ix = np.meshgrid(np.arange(ny) - ny // 2, np.arange(nx) - nx // 2, indexing="ij")
    far = np.hypot(ix, iy) > 0.5
    with rsx.Context(nx, ny, nz, 1, 5.0, algorithm=alg) as ctx:
        ctx.set_morphology(torch.from_numpy(M).cuda())
        ctx.set_optical_constants([285.0], K)
        ctx.set_timing(True)
        got = ctx.run(angles)[0].astype(np.float64)
        assert ctx.phase_times()["fftx"][1] > 0  # the planes path
    err = np.linalg.norm((got - ref)[far]) / np.linalg.norm(ref[far])
    assert err <= 2 * 2.0 ** -25 / s, (err, 2.0 ** -25 / s)
