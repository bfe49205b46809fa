"""A launch that the host refuses leaves no error behind.

The library's runtime keeps the last error of a thread until it is read.  A call
that returned ERR_CUDA has reported it: the next call, whose kernels launch,
must not report it again.  The refused launch is one on a stream whose graph
capture has been invalidated (by a synchronisation of the stream in it)."""
import ctypes

import pytest

import inputs

pytestmark = pytest.mark.gpu

RELAXED = 2  # cudaStreamCaptureModeRelaxed


@pytest.fixture(scope="module")
def cudart():
    import torch
    torch.zeros(1, device="cuda")  # the runtime is loaded
    for name in ("libcudart.so.13", "libcudart.so"):
        try:
            L = ctypes.CDLL(name)
            break
        except OSError:
            continue
    else:
        pytest.skip("no CUDA runtime library to load by name")
    L.cudaStreamBeginCapture.argtypes = [ctypes.c_void_p, ctypes.c_int]
    L.cudaStreamSynchronize.argtypes = [ctypes.c_void_p]
    L.cudaStreamEndCapture.argtypes = [ctypes.c_void_p, ctypes.POINTER(ctypes.c_void_p)]
    return L


@pytest.mark.parametrize("kind", ["one launch", "cluster pairs", "2-D"])
def test_refused_launch_is_reported_once(cudart, kind):
    import torch
    from paper_1908_06649_gb300 import _build
    _build.build()
    import paper_1908_06649_gb300 as pkg
    n, batch = 65536, 4
    x = torch.from_numpy(inputs.make("normal", n, batch, seed=11)).cuda()
    out = torch.empty_like(x)
    plan = {"one launch": lambda: pkg.Plan(n, batch, 16, 3),
            "cluster pairs": lambda: pkg.Plan(n, batch, 16, 3, pkg.PLAN_ONE_PASS),
            "2-D": lambda: pkg.Plan2(256, 256, batch, 16, 3)}[kind]()
    stencil = pkg.StencilPlan(300, 4, 16, 3)
    A = torch.randn(300 * 300, device="cuda")
    B = torch.empty_like(A)
    w3 = [[0.0, 0.1, 0.0], [0.15, 0.5, 0.15], [0.0, 0.1, 0.0]]
    want = stencil.apply(A, w3x3=w3).clone()
    good = plan.forward(x).clone()
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    handle = ctypes.c_void_p(s.cuda_stream)
    assert cudart.cudaStreamBeginCapture(handle, RELAXED) == 0
    assert cudart.cudaStreamSynchronize(handle) != 0  # not allowed: invalidates the capture
    cudart.cudaGetLastError()
    try:
        with pytest.raises(pkg.TcuDftError) as e:
            plan.exec(x, out, pkg.FORWARD, stream=s)
        assert e.value.status == pkg.ERR_CUDA
    finally:
        graph = ctypes.c_void_p()
        assert cudart.cudaStreamEndCapture(handle, ctypes.byref(graph)) != 0
        cudart.cudaGetLastError()
    # the next calls: an element-wise kernel first, then pass kernels
    stencil.apply(A, B, w3x3=w3)
    assert torch.equal(B, want)
    plan.exec(x, out, pkg.FORWARD, stream=s)
    plan.check(s)  # waits for s
    assert torch.equal(out, good)
    stencil.check()
    plan.destroy()
    stencil.destroy()
