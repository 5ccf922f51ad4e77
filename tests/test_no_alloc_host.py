"""The coarse solve without allocation creates nothing: what it uses (events, pinned words)
belongs to the context from mrhs_create on. Shown on the sources, no GPU needed."""
import pathlib
import re

CSRC = pathlib.Path(__file__).parent.parent / "paper_1601_03184_gb300" / "csrc"


def body(text, head):
    """the braces' content of the function whose definition starts with head"""
    at = text.index("{", text.index(head))
    depth, end = 0, at
    while True:
        depth += {"{": 1, "}": -1}.get(text[end], 0)
        end += 1
        if depth == 0:
            return text[at:end]


def test_solve_on_a_given_workspace_creates_nothing():
    text = re.sub(r"//[^\n]*", "", (CSRC / "coarse.cu").read_text())
    for head in ("static void coarse_gmres(", "void coarse_solve_ws("):
        assert not re.findall(r"cuda\w*(?:Create|Malloc|HostAlloc)\w*|\bscratch\(|\bdalloc\(", body(text, head)), head
