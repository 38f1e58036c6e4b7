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
