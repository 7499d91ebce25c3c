"""Inline assembly that reads or writes memory, or orders such accesses, has to
say so to the compiler, which otherwise may move it across stores, barriers and
the wait for the preceding kernel, or merge two of them."""
import pathlib
import re

CSRC = pathlib.Path(__file__).resolve().parent.parent / "paper_2108_02054_gb300" / "csrc"
TOUCHES_MEMORY = re.compile(r"\b(ld|st|red|atom|cp|mbarrier|fence|bar|barrier|membar|griddepcontrol)\.")


def asm_statements(text):
    """Each asm statement with its operands, by counting brackets outside of
    string literals."""
    for m in re.finditer(r"\basm\b", text):
        depth, quoted, i = 0, False, text.index("(", m.end())
        start = i
        while True:
            c = text[i]
            if c == '"' and text[i - 1] != "\\":
                quoted = not quoted
            elif not quoted:
                depth += (c == "(") - (c == ")")
                if depth == 0:
                    break
            i += 1
        yield text[m.start():start], text[start:i + 1]


def test_memory_assembly_is_volatile_and_clobbers_memory():
    seen = 0
    for path in sorted(CSRC.glob("*.cu*")):
        code = re.sub(r"//[^\n]*", "", path.read_text())
        for head, body in asm_statements(code):
            if TOUCHES_MEMORY.search(body):
                seen += 1
                assert "volatile" in head and '"memory"' in body, f"{path.name}: {' '.join(body.split())}"
    assert seen > 0
