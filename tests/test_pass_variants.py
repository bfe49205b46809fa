"""GPU parity of the pass variants at the edges of their items: short last
items, one transform, a batch that no item size divides, the shortest other
side.  Bar: per-transform relative L2 <= 1e-5 (3xTF32) / 3e-3 (TF32) against
the fp64 oracle, the bars of the other parity tests."""
import numpy as np
import pytest

import inputs
import oracle
from oracle import grid

pytestmark = pytest.mark.gpu

TOL = {3: 1e-5, 1: 3e-3, 4: 2e-2, 5: 1e-4}


@pytest.fixture(scope="module")
def pkg():
    from paper_1908_06649_gb300 import _build
    _build.build()
    import paper_1908_06649_gb300 as p
    p.lib()
    return p


def _check_1d(pkg, n, batch, r, prec, inverse, seed):
    import torch
    x = inputs.make("normal", n, batch, seed=seed)
    plan = pkg.Plan(n, batch, r, prec)
    xd = torch.from_numpy(x).cuda()
    y = plan.inverse(xd) if inverse else plan.forward(xd)
    plan.check()
    plan.exec(xd, xd, pkg.INVERSE if inverse else pkg.FORWARD)  # in place
    plan.check()
    assert torch.equal(xd, y)
    err = oracle.rel_l2(y.cpu().numpy(), oracle.dft(x, inverse=inverse, threads=8))
    assert np.all(err <= TOL[prec]), "max rel L2 %.3e" % err.max()
    plan.destroy()


# radix 8, three stages on a strided side: items of four warpgroups hold 8
# sub-transforms, so 1, 3, 7 and 9 of them leave a short last item
@pytest.mark.parametrize("n,batch", [(3 * 512, 1), (5 * 512, 2), (7 * 512, 1), (9 * 512, 3),
                                     (15 * 512, 7), (4 * 512, 1), (4 * 512, 5), (2 * 512, 3),
                                     (8 ** 5, 1), (8 ** 6, 1), (8 ** 7, 1)])
@pytest.mark.parametrize("inverse", [False, True])
def test_radix8_team_items(pkg, n, batch, inverse):
    _check_1d(pkg, n, batch, 8, 3, inverse, seed=n % 97)


# column passes of a runtime shape: one, two and three of them, the fewest
# columns an item spans, a two-level twiddle table (2^20 rows), a batch that
# leaves the last items to few warpgroups, every precision
@pytest.mark.parametrize("r,n1,n2,batch,prec", [
    (8, 512, 8, 1, 3), (8, 512, 64, 3, 3), (8, 512, 512, 1, 5), (8, 4096, 8, 2, 3),
    (8, 4096, 64, 1, 4), (8, 8, 512, 3, 5), (16, 16, 256, 7, 5), (16, 256, 16, 3, 4),
    (16, 4096, 16, 2, 3), (16, 4096, 16, 1, 1), (16, 1 << 20, 16, 1, 3), (32, 1024, 32, 1, 5),
    (32, 32768, 32, 1, 4), (32, 32, 1024, 3, 1)])
@pytest.mark.parametrize("inverse", [False, True])
def test_column_passes(pkg, r, n1, n2, batch, prec, inverse):
    import torch
    x = inputs.make("normal", n1 * n2, batch, seed=5).reshape(batch, n1, n2)
    plan = pkg.Plan2(n1, n2, batch, r, prec)
    d = pkg.INVERSE if inverse else pkg.FORWARD
    xd = torch.from_numpy(x).cuda()
    y = plan.exec(xd, None, d)
    plan.check()
    assert torch.equal(plan.exec(xd, xd, d), y)  # in place
    plan.check()
    yh = y.cpu().numpy().reshape(batch, -1)
    ref = grid.dft2(x, inverse=inverse, threads=8).reshape(batch, -1)
    err = np.linalg.norm(yh - ref, axis=1) / np.linalg.norm(ref, axis=1)
    assert err.max() <= TOL[prec]
    plan.destroy()


# a convolution is two transforms and a product: twice the bar of one (the
# spectrum is given in fp32; the product's rounding is far below)
@pytest.mark.parametrize("r,n1,n2,batch,prec", [
    (16, 256, 4096, 2, 5), (16, 256, 256, 3, 4), (8, 4096, 8, 3, 3), (8, 64, 4096, 1, 3),
    (32, 1024, 1024, 1, 5), (16, 16, 65536, 2, 3)])
def test_column_passes_conv(pkg, r, n1, n2, batch, prec):
    import torch
    x = inputs.make("uniform", n1 * n2, batch, seed=6).reshape(batch, n1, n2)
    w = inputs.make("normal", n1 * n2, 1, seed=7).reshape(n1, n2)
    plan = pkg.Plan2(n1, n2, batch, r, prec)
    xd, wd = torch.from_numpy(x).cuda(), torch.from_numpy(w).cuda()
    y = plan.conv(xd, wd)
    plan.check()
    assert torch.equal(plan.conv(xd, wd, xd), y)
    plan.check()
    ref = torch.fft.ifft2(torch.fft.fft2(torch.from_numpy(x).cdouble())
                          * torch.from_numpy(w).cdouble()).numpy().reshape(batch, -1)
    err = np.linalg.norm(y.cpu().numpy().reshape(batch, -1) - ref, axis=1)
    assert (err / np.linalg.norm(ref, axis=1)).max() <= 2 * TOL[prec]
    plan.destroy()


# real tiles (3xTF32): every radix and tile size, the smallest grids (less than
# a tile), cut blocks, odd sides (rows on no 8-byte boundary), one step, the
# last step count whose spectrum is evaluated directly and the one after it;
# weights without any symmetry.  Bar: 1e-5 max |A|, the stencil tests' bar (the
# weights have unit sum and are not negative).
@pytest.mark.parametrize("r,side,k", [
    (8, 1, 1), (8, 37, 5), (8, 129, 21), (8, 600, 20), (8, 460, 21), (16, 1, 1), (16, 225, 1),
    (16, 449, 16), (16, 448, 16), (16, 300, 20), (16, 301, 21), (16, 500, 85), (32, 33, 2),
    (32, 1000, 20), (32, 1025, 40)])
def test_real_tiles(pkg, r, side, k):
    import torch
    rng = np.random.default_rng(100 * side + k)
    A = rng.standard_normal((side, side)).astype(np.float32)
    w3 = rng.uniform(0.05, 1.0, (3, 3))
    w3 = (w3 / w3.sum()).astype(np.float32)
    plan = pkg.StencilPlan(side, k, r, 3)
    Ad = torch.from_numpy(A).cuda()
    got = plan.apply(Ad, w3x3=w3.tolist())
    plan.check()
    ref = grid.stencil_direct(A.astype(np.float64), w3.astype(np.float64), k)
    assert np.max(np.abs(got.cpu().numpy() - ref)) <= 1e-5 * np.max(np.abs(A))
    plan.apply(Ad, Ad, w3x3=w3.tolist())  # in place
    plan.check()
    assert torch.equal(Ad, got)
    plan.destroy()


# mixed radix with the q-point sums on the way into a tensor-core pass: whole
# transforms (every q that fits, items that use all, some or one transform's
# sub-transforms of theirs, last items of one), and the strided pass of several
@pytest.mark.parametrize("r,q,k,batch", [
    (16, 2, 2, 5), (16, 3, 2, 1), (16, 3, 2, 4), (16, 4, 2, 3), (16, 5, 2, 4), (16, 6, 2, 1),
    (16, 7, 2, 2), (16, 8, 2, 3), (16, 9, 2, 1), (16, 11, 2, 2), (16, 14, 2, 1), (16, 15, 2, 3),
    (16, 3, 1, 43), (16, 15, 1, 9), (16, 2, 3, 3), (16, 8, 3, 1), (16, 2, 4, 1), (16, 4, 4, 1),
    (16, 8, 4, 1), (8, 3, 1, 43), (8, 13, 1, 10), (8, 15, 1, 9), (8, 2, 2, 9), (8, 9, 2, 3),
    (8, 12, 2, 2), (8, 15, 2, 1), (8, 2, 3, 5), (8, 3, 3, 3), (8, 7, 3, 1), (8, 10, 3, 1),
    (8, 2, 4, 3), (8, 4, 4, 1), (32, 3, 1, 43), (32, 14, 1, 10), (32, 2, 2, 3), (32, 3, 2, 2),
    (32, 4, 2, 1), (32, 5, 2, 1), (32, 16, 2, 1), (32, 2, 3, 1), (32, 8, 3, 1), (32, 16, 3, 1)])
@pytest.mark.parametrize("prec,inverse", [(3, False), (3, True), (1, False)])
def test_mixed_on_the_way_in(pkg, r, q, k, batch, prec, inverse):
    _check_1d(pkg, q * r ** k, batch, r, prec, inverse, seed=q + k)


def test_launches_beside_one_another(pkg):
    # pass kernels are set up while the kernel before them runs: a chain of
    # calls that read and overwrite what the last ones wrote, of one to three
    # launches each and with other kernels and table copies between, gives the
    # same bits with and without a synchronisation after every call, on the
    # default and on another stream
    import torch
    n, batch = 4096, 32
    x0 = torch.from_numpy(inputs.make("normal", n, batch, seed=3)).cuda().reshape(-1)
    a = pkg.Plan(4096, 32, 16, 3)          # one launch
    b = pkg.Plan(65536, 2, 16, 3)          # two
    c = pkg.Plan(8192, 16, 16, 3)          # q-point sums on the way in, two
    d = pkg.Plan2(64, 64, 32, 8, 3)        # columns and rows
    s = pkg.StencilPlan(512, 3, 16, 3)     # spectrum, three passes
    w3 = [[0.0, 0.1, 0.0], [0.15, 0.5, 0.15], [0.0, 0.1, 0.0]]

    def chain(sync):
        x, y = x0.clone(), torch.empty_like(x0)
        for i in range(6):
            for f in (lambda: a.forward(x, y), lambda: b.inverse(y, y), lambda: c.forward(y, x),
                      lambda: x.mul_(0.5), lambda: d.inverse(x, y),
                      lambda: pkg.exec_noalloc(y, x, 256 if i & 1 else 512, 512 if i & 1 else 256,
                                               16 if i & 1 else 8, 3),
                      lambda: s.apply(torch.view_as_real(x).reshape(-1),
                                      torch.view_as_real(y).reshape(-1), w3x3=w3),
                      lambda: a.inverse(y, x)):
                f()
                if sync:
                    torch.cuda.synchronize()
        torch.cuda.synchronize()
        return x

    ref = chain(True)
    assert torch.isfinite(torch.view_as_real(ref)).all()
    assert torch.equal(chain(False), ref)
    with torch.cuda.stream(torch.cuda.Stream()):
        assert torch.equal(chain(False), ref)
    for p in (a, b, c, d, s):
        p.check()
        p.destroy()
