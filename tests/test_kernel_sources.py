"""Rules of the kernels that no run can show to be kept, read off their sources."""

import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_21271_b200", "csrc")


def source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def test_the_next_kernel_starts_behind_the_allocation_of_tensor_memory():
    """The weight gradient's copy warps do not wait for their CTA.  Were one of them to let the next kernel start, that kernel could
    take the tensor memory which this CTA has still to allocate, and then wait for this kernel."""
    text = source("split_bwd_weight.cu")
    kernel = text[text.index("split_bwd_weight_kernel("):text.index("split_finalize_kernel(")]
    meeting = kernel.index("bar_sync(2, kThreadsSbw)")
    assert kernel.index("tmem_alloc_pair") < meeting
    early = kernel[kernel.index("if (warp == kWarpTmaM || warp == kWarpTmaN) {"):kernel.index("} else if (warp == kWarpMma) {")]
    for part in (kernel[:meeting], early):
        assert "grid_handover" not in part and "grid_launch_dependents" not in part
    assert kernel.count("grid_handover()") == 2          # the issuing warp's and the sixteen's


@pytest.mark.parametrize("name", sorted(f for f in os.listdir(CSRC) if f.endswith(".cu")))
def test_whole_warps_arrive_at_the_cluster_barrier(name):
    """barrier.cluster.arrive.aligned is for converged warps: directly in front of each stands a barrier of the warp or of more, as
    roles that one lane runs end there."""
    text = source(name)
    for at in (m.start() for m in re.finditer(r"ptx::cluster_arrive\(\);", text)):
        before = re.sub(r"if\s*(constexpr\s*)?\([^;{}]*\)\s*\{?\s*$", "", text[:at]).rstrip()
        last = re.split(r"[;{}]", before.rstrip(";"))[-1].strip()
        assert re.search(r"__syncwarp\(\)|__syncthreads\(\)|bar_sync\(", last), f"{name}: behind '{last}'"
