"""A refinement whose cooperative launch does not fit gives the same flow, bit for
bit, by a launch per round: a child process refuses cooperative launches (a
library preloaded before the CUDA runtime answers for them)."""

import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

REFUSE = r"""
#define _GNU_SOURCE
#include <cuda_runtime_api.h>
#include <dlfcn.h>
int refused;
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **a) {
    for (unsigned i = 0; i < c->numAttrs; ++i)
        if (c->attrs[i].id == cudaLaunchAttributeCooperative && c->attrs[i].val.cooperative) {
            ++refused;
            return cudaErrorCooperativeLaunchTooLarge;
        }
    cudaError_t (*real)(const cudaLaunchConfig_t *, const void *, void **) =
        (cudaError_t (*)(const cudaLaunchConfig_t *, const void *, void **))dlsym(
            dlopen("libcudart.so.13", RTLD_NOW | RTLD_NOLOAD), "cudaLaunchKernelExC");
    return real(c, f, a);
}
"""

CHILD = """
import sys
sys.path[:0] = [{root!r}, {tests!r}]
import ctypes, numpy as np, torch
from test_gpu_refine import _gpu_refine, _texture
out = []
for H, W, C, it, sor in {frames!r}:
    f0 = np.random.default_rng(3).normal(0, 1.0, (H, W, 2)).astype(np.float32)
    out.append(_gpu_refine(_texture(H, W, 1, C), _texture(H, W, 2, C), f0, iterations=it, sor_iterations=sor))
if {so!r}:
    assert ctypes.c_int.in_dll(ctypes.CDLL({so!r}), "refused").value == len(out)
np.savez({to!r}, *out)
"""

FRAMES = [(64, 80, 3, 2, 30), (131, 255, 1, 2, 4), (436, 1024, 3, 3, 30), (19, 300, 4, 3, 10)]


def test_same_flow_without_cooperative_launches(tmp_path):
    from paper_1501_02565_gb300 import build
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build._nvcc()))), "include")
    so = str(tmp_path / "refuse.so")
    (tmp_path / "refuse.c").write_text(REFUSE)
    subprocess.run(["gcc", "-shared", "-fPIC", "-I", include, "-I", "/usr/local/cuda/include", "-o", so,
                    str(tmp_path / "refuse.c"), "-ldl"], check=True)
    flows = []
    for preload in ("", so):
        to = str(tmp_path / f"flows{len(flows)}.npz")
        code = CHILD.format(root=ROOT, tests=os.path.join(ROOT, "tests"), frames=FRAMES, so=preload, to=to)
        env = dict(os.environ, **({"LD_PRELOAD": preload} if preload else {}))
        p = subprocess.run([sys.executable, "-c", code], env=env, capture_output=True, text=True, timeout=300)
        assert p.returncode == 0, p.stderr
        with np.load(to) as z:
            flows.append([z[k] for k in z.files])
    assert len(flows[0]) == len(FRAMES)
    for a, b in zip(*flows):
        assert np.array_equal(a.view(np.int32), b.view(np.int32))
