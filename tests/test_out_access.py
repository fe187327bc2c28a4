"""Which buffers of the caller the listing kernels store into themselves
(csrc/out_access.h), as a host program: only 16-byte aligned memory of the
context's own device.  Any other buffer -- another device's above all, which a
kernel cannot reach without a peer mapping -- gets its rows by a copy."""
import os
import subprocess

from paper_2003_01527_gb300 import build

PROGRAM = r"""
#include <cstdio>
#include <cstring>
#include "out_access.h"
int main() {
  int type, device, ctx;
  unsigned long long at;
  while (scanf("%d %d %llu %d", &type, &device, &at, &ctx) == 4) {
    cudaPointerAttributes a;
    memset(&a, 0, sizeof(a));
    a.type = (cudaMemoryType)type;
    a.device = device;
    printf("%d\n", (int)gsm::kernels_may_store(a, (const void *)(uintptr_t)at, ctx));
  }
}
"""


def test_only_aligned_memory_of_the_own_device(tmp_path):
    src, exe = tmp_path / "rule.cc", tmp_path / "rule"
    src.write_text(PROGRAM)
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build._nvcc()))), "include")
    subprocess.run(["g++", "-std=c++17", "-I" + build.CSRC, "-I" + build.INCLUDE, "-I" + cuda,
                    str(src), "-o", str(exe)], check=True, capture_output=True)
    unregistered, host, dev, managed = range(4)  # cudaMemoryType
    base = 1 << 40
    cases = [((dev, d, base + off, ctx), d == ctx and off % 16 == 0)
             for d in (0, 1, 3) for ctx in (0, 1, 3) for off in (0, 4, 8, 12, 16, 20, 256)]
    cases += [((t, 0, base, 0), False) for t in (unregistered, host, managed)]
    got = subprocess.run([str(exe)], input="\n".join(" ".join(map(str, c)) for c, _ in cases),
                         check=True, capture_output=True, text=True).stdout.split()
    assert got == [str(int(want)) for _, want in cases]
    # and the listing asks this rule before a kernel is given the buffer
    api = open(os.path.join(build.CSRC, "api.cu")).read()
    wide = api[api.index("const bool wide ="):]
    assert "stores_reach(ctx, out)" in wide[:wide.index(";")]
