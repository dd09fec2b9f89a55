"""Every profiler command that the repository gives leaves the GPU's clocks alone."""
import glob
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
FILES = ["bench.py", "README.md", "DESIGN.md"] + sorted(os.path.relpath(p, ROOT) for p in
                                                        glob.glob(os.path.join(ROOT, "profiles", "*.md")))


@pytest.mark.parametrize("name", FILES)
def test_profiler_commands_keep_the_clocks(name):
    """`ncu` locks the clocks unless it is told not to; a command ends at a blank line or a closing fence."""
    text = open(os.path.join(ROOT, name)).read()
    for m in re.finditer(r"(?<![\w`./-])ncu\s+-(?!i\b).*?(?=\n\s*#?\s*\n|\n```|\Z)", text, flags=re.S):
        assert re.search(r"--clock-control[ =]none", m.group(0)), m.group(0)[:200]
