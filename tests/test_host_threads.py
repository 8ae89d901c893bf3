"""Host state of the C entry points, which callers use from any thread: a value kept
between calls is an atomic or lives behind the set-up mutex (no plain function static)."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2608_30877_gb300", "csrc")


def test_function_statics_are_constant_or_atomic():
    bad = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        for i, line in enumerate(open(path), 1):
            m = re.match(r"\s+static\s+(.*)", line)  # indented: inside a function or type
            if m and not re.match(r"(constexpr|const|std::atomic<|__device__)", m.group(1)):
                bad.append(f"{os.path.basename(path)}:{i}: {line.strip()}")
    assert not bad, bad
