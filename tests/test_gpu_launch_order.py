"""Order of the sweeps' kernels with the caller's (needs a B200): the kernels are launched with programmatic dependencies, which must
not show outside a sweep."""
import numpy as np
import pytest
import torch

import oracle
from paper_2601_12917_b200 import synth, zgr

from helpers import ORACLE_DTYPE, from_double, to_double, to_storage, ulp

pytestmark = pytest.mark.gpu

READER = b"""extern "C" __global__ void reader(const unsigned* w, unsigned* out) {
  const unsigned v = w[threadIdx.x];
  asm volatile("griddepcontrol.wait;" ::: "memory");
  out[threadIdx.x] = v;
}"""


def _checked(r):
    assert int(r[0]) == 0, r[0]
    return r[1] if len(r) > 1 else None


def _early_reader():
    """A kernel that is launched with the programmatic attribute and loads 256 words before its own wait, as kernels do with weights
    that they take for constants."""
    from cuda.bindings import driver, nvrtc
    prog = _checked(nvrtc.nvrtcCreateProgram(READER, b"reader.cu", 0, [], []))
    _checked(nvrtc.nvrtcCompileProgram(prog, 1, [b"--gpu-architecture=sm_100a"]))
    cubin = b" " * _checked(nvrtc.nvrtcGetCUBINSize(prog))
    _checked(nvrtc.nvrtcGetCUBIN(prog, cubin))
    module = _checked(driver.cuModuleLoadData(cubin))
    fn = _checked(driver.cuModuleGetFunction(module, b"reader"))

    def launch(words, out):
        import ctypes
        cfg = driver.CUlaunchConfig()
        cfg.gridDimX = cfg.gridDimY = cfg.gridDimZ = 1
        cfg.blockDimX, cfg.blockDimY, cfg.blockDimZ = 256, 1, 1
        cfg.hStream = driver.CUstream(torch.cuda.current_stream().cuda_stream)
        attr = driver.CUlaunchAttribute()
        attr.id = driver.CUlaunchAttributeID.CU_LAUNCH_ATTRIBUTE_PROGRAMMATIC_STREAM_SERIALIZATION
        attr.value.programmaticStreamSerializationAllowed = 1
        cfg.attrs, cfg.numAttrs = [attr], 1
        _checked(driver.cuLaunchKernelEx(cfg, fn, ((words, out), (ctypes.c_void_p, ctypes.c_void_p)), 0))
    launch.module = module
    return launch


# The last 256 words of the last matrix, i.e. of the work that a sweep comes to last, for every kernel family: TMA-staged in two and in three
# parts (ragged, fp32), tile, CUDA-core, isotropic, the last in one and in two launches a sweep.
@pytest.mark.parametrize("dtype,cols,rank,alpha", [("bfloat16", 4096, 32, 0.5), ("bfloat16", 4098, 16, 0.5), ("float32", 4096, 24, 0.5), ("float32", 4098, 24, 0.5), ("float32", 4096, 4, 0.5),
                                                   ("float16", 4096, 0, 1.0)])
@pytest.mark.parametrize("vector", [False, True])
def test_a_kernel_behind_a_sweep_sees_its_weights(dtype, cols, rank, alpha, vector):
    rows = 16384
    w = [torch.zeros(rows, cols, device="cuda", dtype=getattr(torch, dtype))]
    U = [torch.randn(rows, rank, device="cuda") / rows ** 0.5 if rank else None]
    if vector:
        w.append(torch.zeros(100, device="cuda", dtype=w[0].dtype))
        U.append(None)
    z = zgr.Zgr(w, U, alpha, 1e-3, zgr.SCALE_UNIT, 16)
    launch = _early_reader()
    words = w[0].view(torch.int32).view(-1)[-256:]
    out = torch.zeros(256, device="cuda", dtype=torch.int32)
    for i in range(8):
        seed = i // 2 + 1
        if i % 2 == 0:
            z.perturb(seed, 1.0)
        else:
            z.restore_update(seed, 2.0, 1.0, 1e-3)
        launch(words.data_ptr(), out.data_ptr())
        torch.cuda.synchronize()
        assert torch.equal(out, words), f"sweep {i}"
    assert z.device_status() == 0


# One buffer listed twice, as a matrix with a subspace and as a vector without one (or as matrices of two ranks): the kernel
# families run one after the other, so both perturbations arrive.  c z is several times the weights: a lost one shows.
@pytest.mark.parametrize("dtype,rows,cols,ranks", [("f32", 96, 256, (4, 0)), ("bf16", 96, 256, (8, 0)), ("bf16", 256, 1024, (32, 0)), ("bf16", 250, 1025, (16, 0)),
                                                   ("f32", 256, 1024, (4, 8)), ("f32", 256, 1024, (24, 0)), ("f16", 2048, 1032, (16, 8))])
def test_storage_shared_by_two_kernel_families(dtype, rows, cols, ranks):
    ot = ORACLE_DTYPE[dtype]
    w = from_double(oracle.round_to(synth.weights_host(synth.TensorSpec("t", rows, cols, 0), 1).ravel(), ot), dtype, (rows, cols), "cuda")
    views = [w, w if ranks[1] else w.view(-1)]
    U = [torch.from_numpy(synth.subspace(rows, r, 5 + r)).cuda() if r else None for r in ranks]
    z = zgr.Zgr(views, U, 0.5, 1e-3, zgr.SCALE_UNIT, 16)
    a, b = z.scalars()
    for seed, c in ((1, 0.1), (1, -0.2), (2, 0.15)):
        theta = to_storage(w)
        for l, r in enumerate(ranks):
            m, n = (rows, cols) if r else (1, rows * cols)
            t = oracle.OracleTensor(theta=theta, rows=m, cols=n, dtype=ot, U=None if U[l] is None else U[l].cpu().numpy(), q=None, scale=None, zero=None)
            oracle.sweep_tensor(t, seed, l, 16, a, b, c)
            theta = t.theta
        z.sweep_multi([seed], [c])
        torch.cuda.synchronize()
        exp, got = oracle.decode(theta, ot), to_double(w)
        # per sweep 1 ulp of the largest operand (16 bits) or 1e-6 of the largest weight (fp32), as in helpers.check_sweep; two sweeps
        allowed = 2e-6 * np.abs(exp).max() if dtype == "f32" else 2 * ulp(np.full(1, np.abs(exp).max()), dtype)[0]
        assert np.abs(got - exp).max() <= allowed
    assert z.device_status() == 0
