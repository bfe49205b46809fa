"""GPU parity of the one-stage whole transforms (n = 8, 16, 32), whose outputs
leave in 16-byte stores: one transform, a short last item, more items than one
round of the GPU, every precision, in place, on the smallest alignment that is
accepted (16 bytes), and the values around the output left alone.  Bars: the ones
of the other parity tests, against the fp64 oracle."""
import numpy as np
import pytest

import inputs
import oracle

pytestmark = pytest.mark.gpu

TOL = {3: 1e-5, 1: 3e-3, 4: 2e-2, 5: 1e-4}


@pytest.mark.parametrize("r", [8, 16, 32])
@pytest.mark.parametrize("prec", [3, 1, 4, 5])
@pytest.mark.parametrize("batch,inverse", [(1, False), (127, True), (129, False), (200003, True)])
def test_one_stage(r, prec, batch, inverse):
    import torch
    from paper_1908_06649_gb300 import _build
    _build.build()
    import paper_1908_06649_gb300 as pkg
    d = pkg.INVERSE if inverse else pkg.FORWARD
    x = inputs.make("normal", r, batch, seed=r + batch)
    want = oracle.dft(x, inverse=inverse, threads=8)
    # two values (16 bytes) into a buffer, two more behind
    buf = torch.full((batch * r + 4,), 7.0, dtype=torch.complex64, device="cuda")
    out = buf[2:-2]
    assert out.data_ptr() % 32 == 16
    xd = torch.from_numpy(x).cuda().reshape(-1)
    plan = pkg.Plan(r, batch, r, prec)
    plan.exec(xd, out, d)
    plan.check()
    assert np.all(oracle.rel_l2(out.cpu().numpy().reshape(batch, r), want) <= TOL[prec])
    assert torch.all(buf[:2] == 7.0) and torch.all(buf[-2:] == 7.0)
    plan.exec(xd, xd, d)  # in place
    plan.check()
    assert torch.equal(xd, out)
    plan.destroy()
    if prec in (1, 3):
        x2 = torch.from_numpy(x).cuda().reshape(-1)
        assert torch.equal(pkg.exec_noalloc(x2, torch.empty_like(x2), r, batch, r, prec, d), out)


@pytest.mark.parametrize("r,n1", [(8, 512), (16, 256), (32, 1024)])
def test_one_stage_rows(r, n1):
    # rows of one stage in a 2-D transform and in a convolution with a delta
    import torch
    import paper_1908_06649_gb300 as pkg
    x = inputs.make("normal", n1 * r, 3, seed=2).reshape(3, n1, r)
    plan = pkg.Plan2(n1, r, 3, r, 3)
    xd = torch.from_numpy(x).cuda()
    ref = torch.fft.fft2(torch.from_numpy(x).cdouble()).numpy().reshape(3, -1)
    y = plan.exec(xd).cpu().numpy().reshape(3, -1)
    plan.check()
    assert (np.linalg.norm(y - ref, axis=1) / np.linalg.norm(ref, axis=1)).max() <= TOL[3]
    delta = torch.zeros(n1 * r, dtype=torch.complex64, device="cuda")
    delta[0] = 1.0
    one = pkg.Plan2(n1, r, 1, r, 3)
    z = plan.conv(xd, one.exec(delta)).cpu().numpy().reshape(3, -1)
    plan.check()
    x = x.reshape(3, -1)
    assert (np.linalg.norm(z - x, axis=1) / np.linalg.norm(x, axis=1)).max() <= 2 * TOL[3]
    plan.destroy()
    one.destroy()
