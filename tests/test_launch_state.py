"""The launch code keeps nothing that host threads with contexts of their own
share and write: no variables with static storage but constants and the
per-thread message of a failed creation."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1206_0389_gb300", "csrc")
ALLOWED = ("static const ", "static constexpr ", "thread_local ")


def test_no_shared_host_variables():
    found = []
    for name in sorted(os.listdir(CSRC)):
        if not name.endswith((".cu", ".cuh", ".cpp", ".h")):
            continue
        with open(os.path.join(CSRC, name)) as f:
            text = re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", f.read(), flags=re.S))
        for line in text.splitlines():
            s = line.strip()
            # a variable: no parameter list before its initialiser, and not on the device
            if re.match(r"static\s", s) and "(" not in s.split("=")[0] and "__device__" not in s \
                    and not s.startswith(ALLOWED):
                found.append("%s: %s" % (name, s))
    assert not found, found
