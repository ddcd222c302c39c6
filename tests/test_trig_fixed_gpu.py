"""FP64 sine and cosine of the joint angle, seen through a one-link pendulum of unit
mass and length: under a unit base acceleration along z its torque is sin q, along y
cos q (closed form). Both the lane-parallel kernel (small batch) and the serial one.

Bar: 4 x 2^-53 absolute. The angle's reduction and the polynomials are within one ulp
(at most 2^-53 below 1), the one-link recursion multiplies by a few constants of 0 or
1 and adds one product, a rounding each.
"""
import numpy as np
import pytest

import chaingen

pytestmark = pytest.mark.gpu


def angles():
    rng = np.random.default_rng(5)
    half_turns = rng.integers(-1000, 1000, 2000) * (np.pi / 2)
    return np.concatenate([
        rng.uniform(-np.pi, np.pi, 6000), rng.uniform(-1e5, 1e5, 2000),
        rng.uniform(-2.0 ** 30, 2.0 ** 30, 1000), rng.uniform(-1e12, 1e12, 200),  # library beyond 2^30
        half_turns, half_turns + rng.standard_normal(2000) * 2.0 ** -rng.integers(1, 60, 2000),
        2.0 ** -np.arange(0.0, 70.0), [0.0, np.pi / 4, -np.pi / 4, np.nextafter(2.0 ** 30, 0), 2.0 ** 30]])


@pytest.mark.parametrize("small", [True, False])
def test_pendulum_gives_sine_and_cosine(cuda_lib, small):
    import torch

    q = angles()
    if small:
        q = q[:: max(1, len(q) // 1000)]
    model = cuda_lib.Model(chaingen.pendulum(1.0, 1.0))
    x = torch.from_numpy(q).cuda()[:, None].contiguous()
    z = torch.zeros_like(x)
    for axis, f in ((2, np.sin), (1, np.cos)):
        base = np.zeros(18)
        base[6 + axis] = 1.0
        tau = cuda_lib.rnea(model, x, z, z, base=base).cpu().numpy()[:, 0]
        sign = np.sign(tau[0] * f(q[0]))  # the joint's orientation
        err = np.abs(sign * tau - f(q))
        assert err.max() <= 4 * 2.0 ** -53, (axis, q[err.argmax()], err.max())


def test_non_finite_angles_stay_non_finite(cuda_lib):
    import torch

    model = cuda_lib.Model(chaingen.pendulum(1.0, 1.0))
    x = torch.tensor([[np.inf], [-np.inf], [np.nan]], dtype=torch.float64, device="cuda")
    z = torch.zeros_like(x)
    assert torch.isnan(cuda_lib.rnea(model, x, z, z)).all()
