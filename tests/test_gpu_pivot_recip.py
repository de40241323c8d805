"""The reciprocal of a pivot in the Cholesky-inverse kernels against FP64 division, over every exponent
of a positive pivot (the outermost ones take the division itself) and mantissas at both ends."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def test_against_division(cuda):
    from paper_1007_4400_gb300 import gevp
    rng = np.random.default_rng(31)
    mant = np.concatenate([rng.uniform(1, 2, 500), 1 + np.arange(8) * 2.0 ** -52, 2 - np.arange(1, 9) * 2.0 ** -52])
    v = np.ldexp(mant[:, None], np.arange(-1021, 1022)[None, :]).ravel()
    r = gevp.probe_recip(torch.from_numpy(v).to(cuda)).cpu().numpy()
    # e^3 with |e| < 2^-19 and the roundings of the step: half an ulp of the sum, 2^-53 |e| of e
    assert np.all(np.abs(r * v - 1) <= 2.0 ** -52 + 2.0 ** -53)   # (the check's own product rounds too)
    exact = 1 / v
    ulp = np.spacing(np.minimum(exact, np.finfo(float).max / 2))
    assert np.all(np.abs(r - exact) <= ulp)
