"""Order inside kernels that hold tensor memory and let the next kernel start
under them: a CTA of the next kernel may allocate before it waits, so columns
that a CTA of this one still waits for must not be up for the taking.  Read
from the source, since a kernel that breaks the rule hangs the GPU only when
the launches race."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_2406_17782_gb300", "csrc")


def kernels():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        text = re.sub(r"__launch_bounds__\([^)]*\)", "", text)
        for m in re.finditer(r"__global__[^;{]*?(\w+)\([^;{]*\)\s*\{", text):
            depth, at = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(text[at], 0)
                at += 1
            yield m.group(1), text[m.end():at]


def test_dependents_start_once_tensor_memory_is_held():
    seen = []
    for name, body in kernels():
        if "tmem_alloc(" not in body or "grid_dependents_launch()" not in body:
            continue
        seen.append(name)
        alloc = body.index("tmem_alloc(")
        held = re.compile(r"__syncthreads\(\)|sync_all\(\)").search(body, alloc).start()
        assert body.index("grid_dependents_launch()") > held, name
    assert {"decoder_tc_kernel", "train_tc_kernel"} <= set(seen)
