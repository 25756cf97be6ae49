"""Kernels that may start while the one before them in the stream still runs do
not read that kernel's output through the read-only path (``__ldg``), whose data
must not change during the kernel."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1401_7457_gb300", "csrc")
# What an early kernel may read so: the reads' descriptors (written before any
# kernel of the chain), and what its other instantiation alone reads.
ALLOWED = {"onesweep.cuh": r"a\.R\.desc |p\)", "k_emit.cu": r"p \+ q\)"}


def test_no_read_only_loads_of_the_last_kernels_output():
    seen = set()
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        name = os.path.basename(path)
        code = re.sub(r"//.*", "", open(path).read())
        if "grid_dependency_wait();" not in code:
            continue
        seen.add(name)
        head, *kernels = code.split("__global__")  # (helpers stand before the first kernel)
        for part in [head] + [k for k in kernels if "grid_dependency_wait();" in k]:
            for m in re.finditer(r"__ldg\(", part):
                rest = part[m.end():m.end() + 40]
                assert name in ALLOWED and re.match(ALLOWED[name], rest), f"{name}: __ldg({rest}"
    assert {"onesweep.cuh", "k_emit.cu", "k_group.cu", "k_merge.cu"} <= seen
    sort = open(os.path.join(CSRC, "onesweep.cuh")).read()
    assert "return EARLY ? __ldcg(p) : __ldg(p);" in sort
    emit = open(os.path.join(CSRC, "k_emit.cu")).read()
    assert "launch_after(a.id_bytes == 4 &&" in emit  # (64-bit ids, read so, are emitted by a plain launch)
