"""Host side of the launches, by the sources (CPU): a kernel's limit of dynamic shared
memory belongs to the kernel, not to a launch, so that a limit of an object's own size
would refuse another thread's larger launch.  It is set to one value per kernel, where
objects are made."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2012_00881_gb300", "csrc")


def _sources():
    for f in sorted(os.listdir(CSRC)):
        with open(os.path.join(CSRC, f)) as h:
            yield f, h.read()


def test_shared_memory_limits_are_one_value_per_kernel():
    for f, s in _sources():
        for m in re.finditer(r"cudaFuncAttributeMaxDynamicSharedMemorySize,\s*([^;]*?)\)+;", s):
            value = re.sub(r"\(int\)|[()\s]", "", m.group(1))
            assert value in ("most", "kStageSmemMax"), (f, m.group(0))
