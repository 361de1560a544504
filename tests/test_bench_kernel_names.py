"""The benchmark names the kernel that runs and digests the sources of every kernel of its
family (host only)."""
import os

import bench

CSRC = os.path.join(bench.ROOT, "paper_0901_1024_gb300", "csrc")


def test_names_are_kernels_of_the_sources():
    for N in range(1, 10):
        for tc in (False, True) if N <= 7 else (False,):
            name = bench.kernel_name(N, tc).split("<")[0]
            hit = [f for f in bench.KERNEL_SOURCES[bench.kernel_family(N, tc)]
                   if f" {name}(" in open(os.path.join(CSRC, f)).read()
                   or f"\n{name}(" in open(os.path.join(CSRC, f)).read()]
            assert hit, (N, tc, name)
    assert bench.kernel_name(1, False).startswith("direct_stage_kernel")
    assert [bench.kernel_name(N, False).split("<")[0] for N in (8, 9)] == ["stage_wide_kernel"] * 2
    assert bench.kernel_name(4, True) == "tc_stage_kernel<N=4,RK> (tcgen05, FP16x3 split)"
    assert bench.kernel_name(6, True).startswith("tt_stage_kernel<N=6,RK>")
