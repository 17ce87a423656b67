"""The merge kernel for head dim 128 shares the block's registers out anew among
its warpgroups.  What the block has is what the compiler assigned it, which the
launch bounds cap and do not promise: a build with fewer would wait for
registers without end.  The library refuses such a build at run time; this
compiles the kernel and says so earlier."""
import os
import re
import subprocess


def test_compiler_assigns_the_registers_that_are_shared_out(stlib):
    from paper_2608_13667_gb300 import _build
    src = os.path.join(_build.CSRC, "merge_tc.cu")
    with open(src) as f:
        code = f.read()
    soft, other = map(int, re.search(r"kSoftRegs = (\d+), kOtherRegs = (\d+);", code).groups())
    r = subprocess.run([_build._nvcc(), "-c", src, "-o", os.devnull, "-O3", "-std=c++17", "-I", _build.INCLUDE,
                        "--expt-relaxed-constexpr", "-Xptxas", "-v"] + _build.ARCH, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    out = r.stdout + r.stderr
    # merge_pair_kernel<128, false, *>
    used = re.findall(r"Compiling entry function '\w*merge_pair_kernelILi128ELb0ELb[01]E\w*'.*?Used (\d+) registers",
                      out, re.S)
    assert len(used) == 2, out
    for n in map(int, used):
        assert n >= other and 384 * n >= 256 * soft + 128 * other
