"""Function-local state of the library is safe with several host threads: solves of different
plans run at once, so a static that a call fills in is atomic, constant, a mutex or
thread-local. Checked on the source, since a lost race shows rarely.
"""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2401_12890_gb300", "csrc")
SAFE = r"static (?:constexpr|const |thread_local|std::atomic<|std::mutex|__device__|inline)"


def test_statics_are_thread_safe():
    seen = 0
    for f in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        for line in open(f):
            code = line.split("//")[0].strip()
            # a static variable: ends in an initialiser or a semicolon, not a function's head
            if re.match(r"static\b", code) and re.search(r"[;{=]", code) and \
                    not re.match(r"static[^=;{]*\)", code) and not code.startswith("static_assert"):
                seen += 1
                assert re.match(SAFE, code), (os.path.basename(f), code)
    assert seen >= 6
