"""The global-motion fit on any number of blocks. Its blocks wait for one another, so at
most as many as are resident at once are launched: fewer than the 64 parts of the sums
where a process may use only some of the SMs. The parts and the order of their sums do
not depend on it, so neither do the results: the kernel is compiled here with a launch
that takes the number of blocks, and every number gives the same bits."""
import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "gm.cu"
extern "C" int fit(int blocks, const float* pts, int stride, const float* flow, const uint8_t* status, int n, int iters,
                   double c0, double c_min, double* state, double* partial, unsigned* dev_status)
{
    if (blocks < 1 || blocks > kParts) return DGF_ERR_ARG;
    gm_init_kernel<<<1, 1>>>(state);
    void* args[] = {&pts, &stride, &flow, &status, &n, &iters, &c0, &c_min, &state, &partial, &dev_status};
    if (cudaLaunchCooperativeKernel((const void*)gm_fit_kernel, dim3(blocks), dim3(kPartThreads), args, 0, 0) != cudaSuccess)
        return DGF_ERR_CUDA;
    return cudaDeviceSynchronize() == cudaSuccess ? DGF_OK : DGF_ERR_CUDA;
}
// A launch on more blocks than fit the device, which the runtime refuses: the status, and that of a check afterwards.
extern "C" void refused(int* out)
{
    int n = 0, stride = 1, iters = 1;
    double c0 = 1.0, c_min = 1.0;
    void* null = nullptr;
    void* args[] = {&null, &stride, &null, &null, &n, &iters, &c0, &c_min, &null, &null, &null};
    out[0] = dgf::launch_cooperative((const void*)gm_fit_kernel, 1u << 20, dim3(kPartThreads), args, 0);
    out[1] = dgf::launch_status();
    out[2] = dgf::launch_cooperative((const void*)gm_fit_kernel, 0, dim3(kPartThreads), args, 0);
    out[3] = dgf::launch_status();
}
extern "C" size_t partial_bytes() { return kPartialBytes; }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1901_09971_gb300 as dgf
    from paper_1901_09971_gb300 import build
    dgf.load()
    d = tmp_path_factory.mktemp("gm")
    (d / "t.cu").write_text(SOURCE)
    out = str(d / "t.so")
    subprocess.run([build._nvcc(), *build.ARCH, *build.NVCC_FLAGS, "-shared", str(d / "t.cu"), build.LIB, "-Xlinker", "-rpath",
                    "-Xlinker", os.path.dirname(build.LIB), "-o", out], check=True, capture_output=True)
    lib = ctypes.CDLL(out)
    lib.partial_bytes.restype = ctypes.c_size_t
    return lib


@pytest.fixture(scope="module")
def fit(lib):
    def run(blocks, pts, stride, flow, status, n, iters):
        state = torch.zeros(32, dtype=torch.float64, device="cuda")
        partial = torch.full((lib.partial_bytes() // 8,), float("nan"), dtype=torch.float64, device="cuda")
        word = torch.zeros(1, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        ptr = lambda t: ctypes.c_void_p(t.data_ptr())
        rc = lib.fit(blocks, ptr(pts), stride, ptr(flow), ptr(status), n, iters, ctypes.c_double(32.0), ctypes.c_double(2.0),
                     ptr(state), ptr(partial), ptr(word))
        assert rc == 0 and int(word) == 0
        return state[:7].cpu().numpy()  # the affine, then the flags: fitted, go on

    return run


@pytest.mark.parametrize("n", [3, 255, 257, 5000, 16384, 40001])
def test_any_number_of_blocks_gives_the_same_fit(fit, n):
    g = torch.Generator(device="cuda").manual_seed(n)
    stride, iters = 3, 8
    pts = torch.rand((n * stride, 2), device="cuda", generator=g) * 1000
    p = pts[::stride]
    flow = torch.stack([0.01 * p[:, 0] - 0.02 * p[:, 1] + 3, 0.03 * p[:, 0] - 1], 1)
    flow = (flow + 0.3 * torch.randn((n, 2), device="cuda", generator=g)).contiguous()
    flow[::7] += 40  # outliers
    status = (torch.rand(n, device="cuda", generator=g) < 0.1).to(torch.uint8)
    if n == 3:
        status.zero_()
    ref = fit(64, pts, stride, flow, status, n, iters)
    assert np.isfinite(ref[:6]).all() and ref[6:].view(np.int32)[0] == 1
    for blocks in (63, 32, 17, 8, 3, 2, 1):
        np.testing.assert_array_equal(fit(blocks, pts, stride, flow, status, n, iters).view(np.uint64), ref.view(np.uint64))


def test_a_refused_launch_does_not_fail_the_next_call(lib):
    out = (ctypes.c_int * 4)()
    lib.refused(out)
    assert out[0] != 0 and out[1] == 0 and out[2] != 0 and out[3] == 0
