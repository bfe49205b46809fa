"""Rounding of the q-point sums of mixed-radix transforms on the GPU (3xTF32).

Sums that factor are formed in two steps.  They must be no less exact than sums
straight from the definition, whose error for these inputs, against fp64
transforms, was measured with the q-point pass as a launch of its own; where
single roundings fall moves it by a few thousandths, so the bar is 0.5 % above."""
import numpy as np
import pytest

import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r,q,k,forward,inverse", [
    (8, 6, 1, 1.8961e-07, 2.9204e-07), (8, 9, 1, 1.9166e-07, 2.9856e-07),
    (8, 6, 2, 3.2596e-07, 4.2890e-07), (16, 6, 1, 2.1962e-07, 3.0481e-07),
    (16, 9, 1, 2.2140e-07, 2.9536e-07), (16, 6, 2, 3.7786e-07, 4.6235e-07),
    (16, 9, 2, 3.8140e-07, 4.5669e-07), (16, 12, 2, 3.8181e-07, 4.6605e-07),
    (32, 6, 1, 2.7057e-07, 3.5717e-07), (32, 9, 1, 2.7254e-07, 3.3635e-07)])
def test_sums_are_as_exact_as_from_the_definition(r, q, k, forward, inverse):
    import torch
    from paper_1908_06649_gb300 import _build
    _build.build()
    import paper_1908_06649_gb300 as pkg
    n = q * r ** k
    batch = (1 << 21) // n
    x = inputs.make("normal", n, batch, seed=q)
    plan = pkg.Plan(n, batch, r, 3)
    for d, bar in ((pkg.FORWARD, forward), (pkg.INVERSE, inverse)):
        y = plan.exec(torch.from_numpy(x).cuda(), None, d)
        plan.check()
        f = np.fft.fft if d == pkg.FORWARD else np.fft.ifft
        want = f(x.astype(np.complex128), axis=1)
        err = np.linalg.norm(y.cpu().numpy() - want) / np.linalg.norm(want)
        assert err <= 1.005 * bar, "%.4e, from the definition %.4e" % (err, bar)
    plan.destroy()
