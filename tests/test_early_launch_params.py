"""Kernels that may begin while the launch before them runs (they wait in
nr_after_previous) take no __restrict__ pointer to const to what that launch
writes: such loads may use the read-only path, which holds only for data that
nobody writes in the kernel's lifetime."""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
KERNEL = re.compile(r"__global__[^;{]*?\b(\w+_kernel)\s*\(([^{;]*)\)\s*\{(.*?)\n\}\n", re.S)
# what a kernel of a search writes for the next one
HANDED_ON = {"logits", "codes", "nprobe", "x", "seg", "nL", "slen"}


def test_handed_on_buffers_are_not_restrict():
    seen = set()
    for f in glob.glob(os.path.join(ROOT, "paper_2608_15438_gb300", "csrc", "*.cu")):
        for name, params, body in KERNEL.findall(open(f).read()):
            if "nr_after_previous()" not in body:
                continue
            seen.add(name)
            const = re.findall(r"const\s+\w+\s*\*\s*__restrict__\s+(\w+)", params)
            assert not HANDED_ON & set(const), (name, const)
    assert seen == {"route_block_kernel", "select_kernel", "refine_spans_kernel", "encode_layer_kernel"}
