"""A launch attribute without which a kernel cannot run belongs to the function on one device: it may not
hang on a process-wide flag, which the first device's context would set for all, and its result counts.
Read from the sources, since one GPU shows neither."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2302_12727_gb300", "csrc")


def test_shared_memory_limits_are_asked_for_per_context():
    found = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = open(path).read()
        for m in re.finditer(r"cudaFuncAttributeMaxDynamicSharedMemorySize", text):
            found += 1
            call = text.rindex("cudaFuncSetAttribute", 0, m.start())
            statement = text[max(text.rfind(c, 0, call) for c in ";{}") + 1:call]
            assert "=" in statement, f"{os.path.basename(path)}: the result is dropped"
            body = text[text.rindex("\n}\n", 0, call):call]      # from the end of the function before
            assert not re.search(r"\bstatic\s+(bool|int|std::once_flag)\s+\w+\s*(=|;)", body), \
                f"{os.path.basename(path)}: a process-wide flag guards it"
    assert found
