"""A kernel that the caller launches behind a step as its programmatic dependent does not start while the
step still writes weights: only launches that have a dependent of the step's own release it early."""
import ctypes
import subprocess

import pytest
import torch

from paper_2607_19058_gb300 import skewadam as S

pytestmark = pytest.mark.gpu

# One thread takes the time when it starts and when the launch before it is complete.
SRC = r"""
#include <cuda_runtime.h>
__device__ unsigned long long now() { unsigned long long t; asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t)); return t; }
__global__ void k_stamp(unsigned long long *out) {
    out[0] = now();
    asm volatile("griddepcontrol.wait;" ::: "memory");
    out[1] = now();
}
extern "C" int stamp(void *out, void *stream) {
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = cfg.blockDim = dim3(1);
    cfg.stream = (cudaStream_t)stream;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return (int)cudaLaunchKernelEx(&cfg, k_stamp, (unsigned long long *)out);
}
"""


@pytest.fixture(scope="module")
def stamp(tmp_path_factory):
    from paper_2607_19058_gb300 import _build
    _build.build()
    d = tmp_path_factory.mktemp("stamp")
    (d / "stamp.cu").write_text(SRC)
    subprocess.check_call([_build.nvcc(), "-O2", "-Xcompiler", "-fPIC", "-shared", *_build.ARCH, str(d / "stamp.cu"),
                           "-o", str(d / "libstamp.so")])
    lib = ctypes.CDLL(str(d / "libstamp.so"))
    lib.stamp.argtypes = [ctypes.c_void_p, ctypes.c_void_p]
    return lib.stamp


# the last launch: k_apply_rows (2 waves of half tiles of 512 KB, 70 us each), k_apply (2 waves of strip tiles)
@pytest.mark.parametrize("shape", [(38912, 4096), (9728, 8200)], ids=["k_apply_rows", "k_apply"])
def test_last_launch_releases_nothing_early(stamp, shape):
    g = torch.empty(shape, device="cuda").normal_(0, 1e-3).to(torch.bfloat16)
    w = torch.zeros_like(g)
    opt = S.SkewAdam([(w, g, S.TIER_EXPERT)], S.hparams(eps=1e-30))
    out = torch.zeros(2, dtype=torch.int64, device="cuda")
    waited = []
    for t in range(1, 12):
        opt.step(t, 1e-3, 7)
        assert stamp(out.data_ptr(), torch.cuda.current_stream().cuda_stream) == 0
        a, b = out.tolist()
        waited.append((b - a) / 1e3)
    opt.close()
    print(shape, "us from start to completion:", sorted(waited))
    assert sorted(waited)[5] < 8.0
