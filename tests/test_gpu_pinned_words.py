"""The objective's scalars when the pinned words for them cannot be had, at first or
at all: a library linked with a cudaMallocHost that fails on request.  They come
through the pageable fallback then, whatever the graph state, and a call never
returns words that its kernels did not write."""
import ctypes
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SHIM = r"""
extern "C" {
int pinned_failures = 0;  // calls that fail from here on
int __real_cudaMallocHost(void** p, unsigned long n);
int __wrap_cudaMallocHost(void** p, unsigned long n) {
    if (pinned_failures > 0) {
        --pinned_failures;
        return 2;  // cudaErrorMemoryAllocation
    }
    return __real_cudaMallocHost(p, n);
}
}
"""


def _link(tmp):
    from paper_1703_02920_gb300 import build
    build.build()
    src, lib = os.path.join(tmp, "shim.cpp"), os.path.join(tmp, "libmemsynth_shim.so")
    with open(src, "w") as f:
        f.write(SHIM)
    objs = [os.path.join(build.OUT_DIR, os.path.splitext(s)[0] + ".o") for s in build.SOURCES]
    subprocess.run([build._nvcc(), *build.ARCH, "-Xcompiler", "-fPIC", "-shared", "-o", lib, src, *objs, "-Xlinker",
                    "--wrap=cudaMallocHost"], check=True, capture_output=True)
    return lib


def _child(lib_path, failures, through_host):
    """Scalars of three images in the same buffers, on a library of its own."""
    sys.path.insert(0, ROOT)
    import numpy as np
    import torch
    from paper_1703_02920_gb300 import build, memsynth as ms, synth as S
    if lib_path:
        build.LIB = lib_path
    lib = ms.load()
    left = ctypes.c_int.in_dll(lib, "pinned_failures") if lib_path else ctypes.c_int(0)
    ds = S.random_problem(64, 400, 5, lam=1.0)
    left.value = failures
    ctx = ms.Context(ds, precision="fp16x3")
    img = torch.empty(ctx.image_shape(), dtype=torch.float32, device="cuda")
    grad = torch.empty_like(img)
    for k in range(4):  # launched, captured, replayed twice
        if k == 3:
            left.value = 0
        img.copy_(torch.from_numpy(ds.truth * np.float32(1.0 + 0.25 * k)))
        if through_host:
            r = ctx.objective_grad_host(img.cpu().numpy())[:3]
        else:
            r = ms.mem_objective_grad(ctx.handle, img, grad, 0)
        print("RESULT", *[float(x).hex() for x in r])


def _run(lib_path, failures, through_host):
    out = subprocess.run([sys.executable, os.path.abspath(__file__), lib_path, str(failures), str(int(through_host))],
                         capture_output=True, text=True, timeout=600, env=dict(os.environ, PYTHONPATH=ROOT))
    assert out.returncode == 0, out.stdout + out.stderr
    rows = [line.split()[1:] for line in out.stdout.splitlines() if line.startswith("RESULT")]
    assert len(rows) == 4
    return rows


@pytest.mark.parametrize("through_host", [False, True], ids=["device", "host"])
def test_scalars_without_pinned_words(tmp_path, through_host):
    lib = _link(str(tmp_path))
    want = _run("", 0, through_host)
    assert len({r[0] for r in want}) == 4  # the images differ
    # none; the first request only; all until the last call
    for failures in (0, 1, 1000):
        assert _run(lib, failures, through_host) == want, failures


if __name__ == "__main__":
    _child(sys.argv[1], int(sys.argv[2]), bool(int(sys.argv[3])))
