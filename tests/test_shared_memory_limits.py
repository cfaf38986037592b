"""The dynamic shared memory a kernel may have is one setting for all plans and threads of a process: it is set to a value that
follows the device or the library's constants, never to one plan's size."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2305_11998_gb300", "csrc")


def test_limits_do_not_follow_a_plan():
    values = []
    for name in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, name)).read()
        values += re.findall(r"cudaFuncAttributeMaxDynamicSharedMemorySize,([^;]*?)\);", text)
    assert len(values) >= 2
    for value in values:
        words = set(re.findall(r"[A-Za-z_]\w*", value)) - {"int", "moment_smem", "fa", "sharedSizeBytes"}
        assert words <= {"kPartSegments", "optin"}, value
