"""The FP64 reciprocal of the z pivots, which is not the correctly rounded division.

With a Helmholtz shift that dwarfs the couplings a constant f gives p = −f/α, formed as one
reciprocal of the pivot and one product (the transforms of two equal values are exact): within
4·2^-53, of which the pivot's sum, the product and the reciprocal (1.01·2^-53 against the
division's 1) take one each, over the exponents that a pivot may have.
"""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_fp64_pivot_reciprocal(lib):
    import torch
    rng = np.random.default_rng(2)
    f = torch.ones((2, 2, 2), dtype=torch.float64, device="cuda")
    for e in np.linspace(70, 990, 47):
        alpha = float(rng.uniform(1, 2) * 2.0 ** int(e))
        plan = lib.Plan(2, 2, 2, 1.0, 1.0, dz=1.0, bcs=("NN", "NN", "DD"), precision="fp64", alpha=alpha)
        p = plan.solve(f).cpu().numpy()
        plan.close()
        assert np.abs(p * alpha + 1.0).max() <= 5 * 2.0 ** -53, alpha  # (one more for the check's product)
