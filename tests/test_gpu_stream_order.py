"""goq_gemm reads its weights in plain stream order, also behind a kernel that lets its dependents start before it has written
anything (programmatic dependent launch)."""
import numpy as np
import pytest
import torch

import synth_inputs as si

pytestmark = pytest.mark.gpu

LATE_COPY = r"""
extern "C" __global__ void late_copy(const uint4* src, uint4* dst, unsigned long long n) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    for (int i = 0; i < 300; ++i) __nanosleep(1000);   // dependents that do not wait run now
    for (unsigned long long i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (unsigned long long)gridDim.x * blockDim.x) dst[i] = src[i];
}
"""


@pytest.fixture(scope="module")
def goq():
    from paper_2605_26092_b200 import build
    build.build()
    from paper_2605_26092_b200 import goq as g
    g.lib()
    assert torch.cuda.is_available()
    return g


@pytest.fixture(scope="module")
def late_copy():
    """late_copy(src, dst): a kernel on the current stream that copies one byte tensor to another, late."""
    cuda = pytest.importorskip("cuda.bindings.driver")
    nvrtc = pytest.importorskip("cuda.bindings.nvrtc")
    torch.zeros(1, device="cuda")

    def ok(r):
        assert int(r[0]) == 0, r[0]
        return r[1] if len(r) == 2 else r[1:]

    prog = ok(nvrtc.nvrtcCreateProgram(LATE_COPY.encode(), b"late_copy.cu", 0, [], []))
    ok(nvrtc.nvrtcCompileProgram(prog, 1, [b"--gpu-architecture=sm_100"]))
    image = b"\0" * ok(nvrtc.nvrtcGetCUBINSize(prog))
    ok(nvrtc.nvrtcGetCUBIN(prog, image))
    kernel = ok(cuda.cuModuleGetFunction(ok(cuda.cuModuleLoadData(image)), b"late_copy"))

    def run(src, dst):
        assert src.nbytes == dst.nbytes and src.nbytes % 16 == 0 and src.data_ptr() % 16 == 0 and dst.data_ptr() % 16 == 0
        args = [np.array([v], dtype=np.uint64) for v in (src.data_ptr(), dst.data_ptr(), src.nbytes // 16)]
        ptrs = np.array([a.ctypes.data for a in args], dtype=np.uint64)
        ok(cuda.cuLaunchKernel(kernel, 16, 1, 1, 256, 1, 1, 0, torch.cuda.current_stream().cuda_stream, ptrs.ctypes.data, 0))
    return run


@pytest.mark.parametrize("n,k,g,b,m,kind", [(512, 512, 64, 3, 8, "bf16"), (512, 512, 128, 4, 16, "bf16"), (1000, 1024, 128, 3, 24, "bf16"),
                                            (1000, 1024, 128, 3, 64, "bf16"), (1000, 1024, 16, 3, 300, "bf16"), (1024, 1024, 64, 2, 2100, "bf16"),
                                            (256, 512, 8, 4, 40, "bf16"), (512, 512, 64, 3, 200, "i8"), (128, 512, 32, 4, 7, "i8"),
                                            (512, 512, 16, 3, 64, "i8"), (512, 512, 64, 3, 64, "requant")])
def test_weights_written_late_by_the_kernel_before(goq, late_copy, n, k, g, b, m, kind):
    """The weight buffer holds one layer; a kernel that is still in flight when goq_gemm is issued overwrites it with another. The
    result is the other layer's, bit for bit, on every path of the dispatch."""
    from tests.gpu_util import dev, pack_weights
    rng = np.random.default_rng(n + m)
    (d, old), (_, new) = (pack_weights(n, k, g, b, *si.random_quantized(n, k, g, b, seed=s)) for s in (1, 2))
    packed = old.clone()
    if kind == "bf16":
        x = dev(si.bf16_activations(m, k, seed=3))
        ws = goq.new_workspace(d, goq.OP_GEMM, m)
        y = torch.zeros((m, n), dtype=torch.float32, device="cuda")

        def call(w):
            goq.gemm(d, w, x, m, goq.BF16, y=y, y_dtype=goq.F32, ws=ws)
    else:
        x = dev(rng.integers(-127, 128, size=(m, k)).astype(np.int8))
        cq = dev(rng.integers(-127, 128, size=(n, k // g, 2)).astype(np.int8))
        sx, sc = torch.ones(m, device="cuda"), torch.ones((n, 2), device="cuda")
        y, amax = torch.zeros((m, n), dtype=torch.float32, device="cuda"), torch.zeros(m, device="cuda")

        def call(w):
            if kind == "i8":
                goq.gemm(d, w, x, m, goq.I8, y=y, y_dtype=goq.F32, sx=sx, cq=cq, sc=sc)
            else:
                goq.gemm_i8_requant(d, w, x, m, sx, cq, sc, y, amax)
    refs = []
    for w in (old, new):
        call(w)
        torch.cuda.synchronize()
        refs.append(y.clone())
    assert not torch.equal(*refs)
    stream = torch.cuda.Stream()
    for _ in range(3):
        packed.copy_(old)
        y.zero_()
        torch.cuda.synchronize()
        with torch.cuda.stream(stream):
            late_copy(new, packed)
            call(packed)
        torch.cuda.synchronize()
        assert torch.equal(y, refs[1])
