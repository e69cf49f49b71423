"""Properties of the CUDA sources that no result shows reliably."""
import re
from pathlib import Path

CSRC = Path(__file__).resolve().parents[1] / "paper_1809_08013_gb300" / "csrc"


def _sources():
    return {f.name: f.read_text() for f in sorted(CSRC.glob("*.cu*"))}


def _asm_statements(text):
    for m in re.finditer(r"\basm\b(?:\s+volatile)?\s*\(", text):
        depth, quoted, k = 1, False, m.end()
        while depth:
            c = text[k]
            if c == '"' and text[k - 1] != "\\":
                quoted = not quoted
            elif not quoted:
                depth += (c == "(") - (c == ")")
            k += 1
        yield text[m.start():k]


def test_asm_that_writes_memory_says_so():
    # without the clobber the compiler may keep, or move across it, ordinary
    # accesses to what the statement stores
    seen = 0
    for name, text in _sources().items():
        for s in _asm_statements(text):
            template = "".join(re.findall(r'"((?:[^"\\]|\\.)*)"', s.split(":")[0]))
            if re.search(r"\b(st|red|atom)\.", template):
                seen += 1
                assert '"memory"' in s, (name, s)
    assert seen > 0


def test_no_launch_needs_the_whole_gpu():
    # a cooperative launch starts only when all its blocks fit at once: contexts
    # that step on streams of their own then wait for one another
    for name, text in _sources().items():
        assert "LaunchCooperative" not in text and "cooperative_groups" not in text, name
