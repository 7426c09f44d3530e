"""Launches that overlap the end of the launch before them: every kernel that may be placed early waits for its predecessor
before anything else, in every block.  Read off the sources, since a block that reads too early gives no error."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2111_06483_b200", "csrc")


def sources():
    return {f: open(os.path.join(CSRC, f)).read() for f in sorted(os.listdir(CSRC)) if f.endswith((".cu", ".cuh"))}


def test_every_early_placed_kernel_waits_first():
    text = sources()
    every = "\n".join(text.values())
    seen = 0
    for f, s in text.items():
        for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\(.*?\)\s*)?(\w+)\(", s):
            name, body = m.group(1), s[s.index("{", m.end()) + 1:]
            if re.search(name + r"(?:<[^;{}]*?>)?\s*<<<", every):
                continue   # launched in stream order
            first = next(line.strip() for line in body.splitlines()
                         if line.strip() and not re.match(r"(?://|constexpr|static_assert|using)", line.strip()))
            assert first == "after_predecessor();", (f, name, first)
            seen += 1
    assert seen >= 15


def test_nothing_else_touches_the_order():
    for f, s in sources().items():
        for at in re.finditer(r"griddepcontrol\.\w+", s):
            line = s[s.rfind("\n", 0, at.start()) + 1:at.start()]
            assert f == "sar_launch.cuh" or line.lstrip().startswith("//"), f
    s = sources()["sar_launch.cuh"]
    assert s.index("griddepcontrol.wait") < s.index("griddepcontrol.launch_dependents") and s.count('"griddepcontrol.') == 2
