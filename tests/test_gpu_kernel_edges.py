"""Kernels at the edges of their ranges: sizes around a tile, a group or a block, and the ends of a
dispatch rule, against the FP64 oracle or against an exact relation."""
import numpy as np
import pytest

from paper_1907_01724_gb300 import api, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [2.0 ** -490, 2.0 ** -300, 2.0 ** 300])
@pytest.mark.parametrize("n", [1, 129])
def test_fp64_potentials_scale_with_the_cavity(n, scale):
    """A cavity scaled by a power of two has its potentials scaled by the inverse (the FP64 pair
    kernel's reciprocal roots at both ends of their range and in their fallback for tiny
    arguments)."""
    rng = np.random.default_rng(190790 + n)
    xyz, q = inputs.uniform_ball(rng, n, 1.0), rng.choice([-1.0, 1.0], n)
    phi = [api.solve(inputs.System(a, 2.0, 80.0, 1.5 / a, 12, 64, a * xyz, q), precision=api.HSMA_FP64).phi
           for a in (1.0, scale)]
    # every operation scales exactly except through the range of exponents: rounding of a few sums
    assert np.linalg.norm(phi[1] * scale - phi[0]) <= 1e-12 * np.linalg.norm(phi[0])
