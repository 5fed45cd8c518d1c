"""Which memory the kernels use where it lies: a host check of the rule (another GPU's
memory and odd addresses are copied), and the copies' results on the GPU."""
import subprocess

import numpy as np
import pytest

from paper_1805_03426_gb300 import build

SRC = r"""
#include <stdio.h>
#include "mr_internal.cuh"
int main()
{
    const int types[] = {cudaMemoryTypeUnregistered, cudaMemoryTypeHost, cudaMemoryTypeDevice, cudaMemoryTypeManaged};
    for (int t : types)
        for (int at = 0; at < 2; ++at)
            for (size_t p : {4096, 4100, 4104}) {
                cudaPointerAttributes a = {};
                a.type = (cudaMemoryType)t;
                a.device = at;
                printf("%d", mr::usable_in_place(a, 1, (const void*)p));
            }
    return 0;
}
"""


def test_rule(tmp_path):
    src, exe = tmp_path / "p.cu", tmp_path / "p"
    src.write_text(SRC)
    subprocess.run([build._nvcc(), *build.ARCH, "-std=c++17", "-I", build.CSRC, "-I", build.ROOT + "/include", "-o", str(exe),
                    str(src)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    # ordinary and pinned host memory; device memory elsewhere and here; managed memory
    assert out == "000000" + "000000" + "000101" + "101101"


def _unaligned(n, dtype):
    """Device memory of n values that starts off their boundary by four bytes: (raw bytes, pointer)."""
    import torch

    raw = torch.zeros(n * np.dtype(dtype).itemsize + 8, dtype=torch.uint8, device="cuda")
    return raw, raw.data_ptr() + 4


@pytest.mark.gpu
@pytest.mark.parametrize("mode,f64", [("fused", False), ("xfused", False), ("stored", False), ("stored", True)])
def test_unaligned_device_faces_are_copied(mode, f64):
    torch = pytest.importorskip("torch")
    import paper_1805_03426_gb300.mr as mr
    from tests.gpu_common import Problem
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    p = Problem(nx=16, ny=8, nz=7, mx=4, my=4, mz=4, gamma=1.5)
    vm = {"stored": mr.MR_VEL_STORED, "fused": mr.MR_VEL_FUSED, "xfused": mr.MR_VEL_XFUSED}[mode]
    dtype = np.float64 if f64 else np.float32
    out = []
    for odd in (False, True):
        h = mr.mr_create(p.mr_config(mr, mr.MR_F64 if f64 else mr.MR_F32, vm))
        keep, ptr = [], []
        for a in (p.U, p.V, p.W):
            raw, q = _unaligned(a.size, np.float64)
            if not odd:
                q -= 4
            off = q - raw.data_ptr()
            raw[off:off + a.nbytes] = torch.from_numpy(np.ascontiguousarray(a).reshape(-1).view(np.uint8).copy()).cuda()
            keep.append(raw)
            ptr.append(q)
        faces = [(h.shapes[k], *_unaligned(int(np.prod(h.shapes[k])), dtype)) for k in ("Us", "Vs", "Ws")]
        dense = [q if odd else q - 4 for _, _, q in faces] if mode == "stored" else [None] * 3
        st = torch.cuda.current_stream().cuda_stream
        mr._check(mr.lib().mr_refine_velocity(h.ptr, *ptr, *dense, st))
        mr.mr_set_scalar(h, torch.from_numpy(p.T0).cuda())
        mr.mr_scalar_step(h, 3)
        T = torch.empty(p.T0.shape, dtype=torch.float64, device="cuda")
        mr.mr_get_scalar(h, T)
        torch.cuda.synchronize()
        got = [T.cpu().numpy()]
        for (shape, raw, q), d in zip(faces, dense):
            if d:
                b = raw.cpu().numpy()[d - raw.data_ptr():][:int(np.prod(shape)) * np.dtype(dtype).itemsize]
                got.append(np.frombuffer(b.tobytes(), dtype).reshape(shape))
        out.append(got)
        h.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b) and np.abs(a).max() > 0
