"""A host buffer is read and written in place by a kernel only where page-locked ranges cover all
of it: the rule itself on the host, and copies to and from partly registered buffers on the GPU."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from tests.conftest import ROOT

RULE = r"""
#include <cstdio>
#include <cstdlib>
#include "host_range.h"
// ranges {start, size, device offset}, then buffers {p, bytes}; prints the address or 0 of each buffer
int main(int argc, char** argv) {
  const int n = atoi(argv[1]);
  char** a = argv + 2;
  auto query = [&](uintptr_t p) {
    icon::HostRange r;
    for (int i = 0; i < n; ++i) {
      const uintptr_t s = strtoull(a[3 * i], 0, 0), z = strtoull(a[3 * i + 1], 0, 0);
      if (p >= s && p < s + z) { r.start = s; r.size = z; r.dev = p + strtoull(a[3 * i + 2], 0, 0); }
    }
    return r;
  };
  for (int i = 2 + 3 * n; i + 1 < argc; i += 2)
    printf("%llu\n", (unsigned long long)icon::mapped_address(strtoull(argv[i], 0, 0), strtoull(argv[i + 1], 0, 0), query));
  return 0;
}
"""


def test_only_buffers_covered_without_a_gap_are_mapped(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    src, exe = tmp_path / "rule.cpp", tmp_path / "rule"
    src.write_text(RULE)
    subprocess.run([cxx, "-std=c++17", "-I", os.path.join(ROOT, "paper_2511_02021_gb300", "csrc"), str(src), "-o",
                    str(exe)], check=True)
    K = 4096
    ranges = [(16 * K, 4 * K, 0), (20 * K, K, 0),            # two registrations side by side
              (32 * K, K, 0), (40 * K, K, 0),                # both ends of a buffer, nothing between
              (64 * K, K, 512 * K), (65 * K, K, 700 * K)]    # side by side, not so on the device
    buffers = {(16 * K, 4 * K): 16 * K, (16 * K + 8, K): 16 * K + 8, (16 * K, 5 * K): 16 * K, (19 * K, 2 * K): 19 * K,
               (16 * K, 5 * K + 8): 0, (15 * K, K): 0, (15 * K, 2 * K): 0,
               (32 * K, 9 * K): 0, (32 * K, K): 32 * K, (40 * K, K): 40 * K,
               (64 * K, K): 576 * K, (64 * K, 2 * K): 0, (8, 8): 0}
    args = [str(len(ranges))] + [str(v) for r in ranges for v in r] + [str(v) for b in buffers for v in b]
    out = subprocess.run([str(exe)] + args, check=True, capture_output=True, text=True).stdout.split()
    assert dict(zip(buffers, map(int, out))) == buffers


@pytest.mark.gpu
@pytest.mark.parametrize("registered", ["ends", "start", "halves", "whole"])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_copies_take_partly_registered_buffers(gpu, precision, registered):
    """Registered at the ends only, at its start only, in two halves, or as a whole: every field,
    a tracer and a decomposed state's field arrive as in pageable memory."""
    import torch
    C = gpu
    N, K = 33, 65536
    cudart = torch.cuda.cudart()
    grid = C.icon_grid_build(2, 2, N)
    st = C.icon_state_init_ex(grid, 3, C.ICON_CASE_JET, noise_K=0.1,
                              precision=C.ICON_MIXED if precision == "mixed" else C.ICON_FP64)
    C.icon_dycore_step(st, 300.0, 5)                         # forms the step-mean fluxes
    dom = C.icon_domain_create(st, 2, 3) if precision == "fp64" else None
    rng = np.random.default_rng(4)

    def buffer(shape):
        n = int(np.prod(shape)) * 8
        raw = np.zeros(n + 2 * K, np.uint8)
        base = (raw.ctypes.data + K - 1) // K * K
        end = base + n // K * K
        assert n >= 4 * K
        parts = {"ends": [(base, K), (end - K, n - (end - K - base))], "start": [(base, K)], "whole": [(base, n)],
                 "halves": [(base, 2 * K), (base + 2 * K, n - 2 * K)]}[registered]
        for p, z in parts:
            assert int(cudart.cudaHostRegister(p, z, 0)) == 0
        o = base - raw.ctypes.data
        return raw[o:o + n].view(np.float64).reshape(shape), [p for p, _ in parts], raw

    try:
        for f in C.FIELDS:
            want = C.icon_state_copy_field(st, grid, N, f)
            buf, regs, raw = buffer(want.shape)
            try:
                assert np.array_equal(C.icon_state_copy_field(st, grid, N, f, buf), want), f
                if f in ("vn", "w", "rho", "theta_v", "exner"):
                    buf[...] = rng.uniform(0.5, 1.5, want.shape).astype(np.float32)
                    C.icon_state_set_field(st, grid, N, f, buf)
                    assert np.array_equal(C.icon_state_copy_field(st, grid, N, f), buf), f
                    C.icon_state_set_field(st, grid, N, f, want)
                    if dom is not None:
                        C._check(C._lib.icon_domain_copy_field(dom, C.FIELDS[f][0], buf.ctypes.data, buf.size))
                        assert np.array_equal(buf, want), f
            finally:
                for p in regs:
                    cudart.cudaHostUnregister(p)
        C.icon_state_add_tracers(st, 1)
        x = rng.uniform(0.0, 1.0, (C.icon_grid_counts(grid)[0], N))
        buf, regs, raw = buffer(x.shape)
        try:
            buf[...] = x
            C.icon_state_set_tracer(st, grid, N, 0, buf)
            assert np.array_equal(C.icon_state_copy_tracer(st, grid, N, 0), x)
            buf[...] = 0.0
            C._check(C._lib.icon_state_copy_tracer(st, 0, buf.ctypes.data, buf.size))
            assert np.array_equal(buf, x)
        finally:
            for p in regs:
                cudart.cudaHostUnregister(p)
    finally:
        if dom is not None:
            C.icon_domain_free(dom)
        C.icon_state_free(st)
        C.icon_grid_free(grid)
