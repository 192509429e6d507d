"""The C-ABI library builds, loads and exports every declared entry point
(CPU only: no compute call is made here)."""
import ctypes
import glob
import os
import re
import shutil

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def declared_functions():
    names = set()
    for h in glob.glob(os.path.join(ROOT, "include", "*.h")):
        text = open(h).read()
        text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
        text = re.sub(r"//[^\n]*", "", text)
        for m in re.finditer(r"\b([a-z_][a-z0-9_]*)\s*\(", text):
            name = m.group(1)
            if name.startswith("schulze_") and not name.endswith("_t"):
                names.add(name)
    return sorted(names)


@pytest.fixture(scope="module")
def lib():
    if shutil.which("nvcc") is None and not os.path.exists("/usr/local/cuda/bin/nvcc"):
        pytest.skip("nvcc not available")
    from paper_2505_12976_gb300 import _build
    path = _build.build()
    return ctypes.CDLL(path)


def test_headers_declare_the_path():
    names = declared_functions()
    for required in ("schulze_tally", "schulze_strongest_paths", "schulze_winners", "schulze_ranking",
                     "schulze_run", "schulze_run_host", "schulze_ctx_create", "schulze_get_status"):
        assert required in names


def test_library_exports_every_declared_symbol(lib):
    missing = [n for n in declared_functions() if not hasattr(lib, n)]
    assert not missing, f"declared but not exported: {missing}"


def test_binding_covers_every_declared_symbol(lib):
    import paper_2505_12976_gb300 as S
    bound = {name for name, _, _ in S.SIGNATURES}
    assert set(declared_functions()) <= bound


def test_strerror_without_gpu(lib):
    lib.schulze_strerror.restype = ctypes.c_char_p
    assert lib.schulze_strerror(0) == b"ok"
    assert b"invalid" in lib.schulze_strerror(-1)


def test_argument_checks_without_gpu(lib):
    """Host-side validation rejects bad arguments before touching CUDA."""
    v = ctypes.c_void_p
    lib.schulze_tally.argtypes = [v, v, ctypes.c_int64, ctypes.c_int32, ctypes.c_int32, v, ctypes.c_uint32, v]
    lib.schulze_ctx_create.argtypes = [ctypes.c_int, ctypes.POINTER(v)]
    assert lib.schulze_tally(None, None, 1, 4, 4, None, 0, None) == -1
    assert lib.schulze_ctx_create(-1, ctypes.byref(v())) == -1
    lib.schulze_set_wait_limit.argtypes = [v, ctypes.c_int64]
    assert lib.schulze_set_wait_limit(None, 1000) == -1


def test_host_call_argument_checks_without_gpu(lib):
    """schulze_run_host: the C entry point rejects a missing context with
    SCHULZE_EINVAL, and the binding rejects ballots of the wrong type or
    layout, both before any CUDA call."""
    v = ctypes.c_void_p
    lib.schulze_run_host.argtypes = [v, v, ctypes.c_int64, ctypes.c_int32, ctypes.c_int32, v, v, ctypes.c_uint32, v]
    buf = (ctypes.c_int32 * 16)()
    assert lib.schulze_run_host(None, ctypes.cast(buf, v), 2, 4, 2, None, None, 0, None) == -1  # no context
    import numpy as np
    import paper_2505_12976_gb300 as S
    with pytest.raises(ValueError):
        S.schulze_run_host(np.zeros((2, 3), np.int64), 4)  # not int32
    with pytest.raises(ValueError):
        S.schulze_run_host(np.zeros((3, 2), np.int32).T, 4)  # not C-contiguous
    import torch
    with pytest.raises(ValueError):
        S.schulze_run_host(torch.zeros((2, 3), dtype=torch.int64), 4)


def test_product_path_has_no_cpu_fallback():
    """The binding refuses to run when the library is missing, and nothing in
    the package imports the oracle."""
    pkg = os.path.join(ROOT, "paper_2505_12976_gb300")
    for f in glob.glob(os.path.join(pkg, "**", "*.py"), recursive=True):
        src = open(f).read()
        assert "import oracle" not in src and "from oracle" not in src, f


def run_probe(tmp_path, text):
    """Compiles host code against the internal header and the library's
    objects, runs it and returns its exit code."""
    import subprocess

    from paper_2505_12976_gb300 import _build
    src, exe = tmp_path / "probe.cu", tmp_path / "probe"
    src.write_text(text)
    subprocess.run([_build._nvcc(), *_build.ARCH, "-std=c++17", "--expt-relaxed-constexpr",
                    "-I", os.path.join(ROOT, "include"), "-I", _build.CSRC, str(src),
                    *sorted(glob.glob(os.path.join(_build.BUILD, "*.o"))), "-o", str(exe)], check=True)
    return subprocess.run([str(exe)]).returncode


ZERO_SPANS_PROBE = r"""
#include "internal.cuh"
// spans with nothing to zero take no place; one too many is reported
int main() {
  using namespace schulze;
  uint32_t w[16] = {};
  ZeroSpans z;
  z.add(nullptr, 4), z.add(w, 0);
  for (int q = 0; q < kZeroSpans; ++q) z.add(w + q, 1);
  for (int q = 0; q < kZeroSpans; ++q)
    if (z.p[q] != w + q || z.words[q] != 1) return 1;
  z.add(nullptr, 4), z.add(w, 0);
  if (z.overflow) return 2;
  z.add(w + kZeroSpans, 1);
  if (!z.overflow) return 3;
  return zero_async(nullptr, z, nullptr) == SCHULZE_EINVAL ? 0 : 4;
}
"""


def test_zero_spans_refuse_one_too_many(lib, tmp_path):
    """A span that finds no place makes the zeroing fail instead of being
    left out (host code: no launch is made)."""
    assert run_probe(tmp_path, ZERO_SPANS_PROBE) == 0


NO_MEMORY_PROBE = r"""
#include <stdlib.h>

#include "internal.cuh"
static bool deny = false;
void* operator new(size_t n) {
#ifndef __CUDA_ARCH__
  if (deny) exit(9);  // an allocation, which could have thrown
#endif
  return malloc(n ? n : 1);
}
void operator delete(void* p) noexcept { free(p); }
void operator delete(void* p, size_t) noexcept { free(p); }
__global__ void some_kernel() {}
// the launch helpers remember what they asked for without allocating, also
// past what they can hold
int main() {
  using namespace schulze;
  schulze_ctx* ctx = new schulze_ctx();
  deny = true;
  const void* fn = reinterpret_cast<const void*>(some_kernel);
  for (int q = 0; q < 200; ++q) {
    raise_smem(ctx, q % 2 ? fn : static_cast<const char*>(fn) + q);
    if (blocks_per_sm(ctx, fn, 32, size_t(q)) < 1) return 2;
    remember(ctx, Residency{fn, 32, size_t(q), 3});
    if (blocks_per_sm(ctx, fn, 32, size_t(q)) != 3) return 3;
  }
  return 0;
}
"""


def test_launch_helpers_do_not_allocate(lib, tmp_path):
    """No exception can leave a C entry from the launch helpers (host code: no
    launch is made)."""
    assert run_probe(tmp_path, NO_MEMORY_PROBE) == 0
