"""The host code builds for the processors that B200s come with: what only x86 has stands behind a test for x86."""

import re
from pathlib import Path

CSRC = Path(__file__).resolve().parent.parent / "paper_1802_04819_b200" / "csrc"


def test_x86_intrinsics_are_guarded():
    for path in sorted(CSRC.iterdir()):
        guards = []
        for number, line in enumerate(path.read_text().splitlines(), 1):
            if re.match(r"\s*#\s*if", line):
                guards.append(line)
            elif re.match(r"\s*#\s*el", line):
                guards[-1] = line
            elif re.match(r"\s*#\s*endif", line):
                guards.pop()
            elif re.search(r"\b_mm\w*\s*\(|\w*mmintrin\.h|\b__builtin_ia32", line):
                assert any("__x86_64__" in g for g in guards), f"{path.name}:{number}: {line.strip()}"
