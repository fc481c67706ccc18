"""A kernel that lets its successor start before its own dependency wait hands on no ordering: what the successor reads before it waits
itself (weights, inputs, regions of the workspace) may still be being written.  In the kernels' source the wait comes first, except in
those that always follow a kernel which has waited and whose successors read nothing of theirs early."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2602_12128_b200", "csrc")
# the reduction, whose predecessor (the fused key side) releases it after its own wait, and the three that wait late behind a reduction
AFTER_ONE_THAT_WAITED = {"tc_reduce_emit_kernel", "tc_readout_kernel", "tc_bwd_key_kernel", "phiq_cta"}


def bodies():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cuh"))):
        if path.endswith("hla_tc_prim.cuh"):
            continue
        text = re.sub(r"//[^\n]*", "", open(path).read())
        heads = [m for m in re.finditer(r"^(?:__global__|__device__)[^;{]*?\b(\w+)\((?=const|CUtensorMap|Dims|float|VmlpPtrs|int|T\b)", text, flags=re.M)]
        for i, m in enumerate(heads):
            yield m.group(1), text[m.start(): heads[i + 1].start() if i + 1 < len(heads) else len(text)]


def test_wait_before_release():
    seen = set()
    for name, body in bodies():
        release = re.search(r"grid_launch_dependents\(\)", body)
        if release:
            seen.add(name)
            if name not in AFTER_ONE_THAT_WAITED:
                wait = re.search(r"grid_dependency_wait\(\)", body)
                assert wait and wait.start() < release.start(), name
    assert AFTER_ONE_THAT_WAITED <= seen and "phik_state_cta" in seen and "tc_causal_forward_kernel" in seen
