"""Host side of the launches, by the sources (CPU): a kernel's limit of dynamic shared
memory belongs to the kernel, not to a launch, so that a limit of an object's own size
would refuse another thread's larger launch.  It is set to one value per kernel, where
objects are made.  And what a kernel reads is copied on the object's own stream: one
that does not wait for the default stream could launch before a copy there has landed
(from pageable memory such a copy returns when it is staged)."""
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


def test_nothing_is_copied_to_the_device_on_the_default_stream():
    for f, s in _sources():
        for m in re.finditer(r"cudaMemcpy\([^;]*;", s):
            assert "HostToDevice" not in m.group(0), (f, m.group(0))
