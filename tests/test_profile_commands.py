"""Every ncu command that a profile summary quotes leaves the GPU's clocks
alone: run as written, ncu without that switch locks them."""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_quoted_ncu_commands_leave_the_clocks():
    seen = 0
    for path in sorted(glob.glob(os.path.join(ROOT, "profiles", "*")) + [os.path.join(ROOT, "DESIGN.md")]):
        text = re.sub(r"\\\n\s*", " ", open(path).read())
        for cmd in re.findall(r"\bncu --?[a-z][^\n`;)]*", text):
            seen += 1
            assert "--clock-control none" in cmd, f"{os.path.basename(path)}: {cmd}"
    assert seen > 0
