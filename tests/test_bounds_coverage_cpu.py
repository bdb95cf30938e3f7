"""What the bounds-checking build checks, on the sources: in the kernels that reach a block's arrays
(the sweep, the sum that ends a stage, the speed and time-step reductions, the halo packing) every
access through one of the arrays' pointers names its bounds (FPK_IN)."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2101_05886_gb300", "csrc")
# pointers to a block's arrays in these files (the caller's state, halo or output, the context's own)
ARRAYS = r"(?:q|qi|q0|qn|qs|qin|kj|fk|out|racc|ra|a|src|qp|q4)"


def _statements(name):
    """The file's statements without comments, from the first kernel on."""
    text = open(os.path.join(CSRC, name)).read()
    text = re.sub(r"//[^\n]*", "", text)
    if name == "sweep.cuh":
        text = text[text.index("fp_sweep(const BlockDev"):text.index("sweep_smem()")]
    return [" ".join(s.split()) for s in re.split(r"[;{}]", text)]


@pytest.mark.parametrize("name", ["sweep.cuh", "stage.cu", "cfl.cu"])
def test_every_access_to_a_blocks_array_names_its_bounds(name):
    bare = []
    statements = _statements(name)
    checked = [m.group(1) for s in statements for m in [re.search(r"\b(\w+) = FPK_IN\(", s)] if m]   # pointers checked as they are made
    for s in statements:
        if any(re.search(rf"\b{p} \+ c\b", s) for p in checked):
            continue
        wide = re.search(r"\b(?:load4|store4|cp_async_\w*el)\(", s) and not re.search(r"\b(?:epb|nsb)\b", s)
        element = re.search(r"\*\s*comp_at\(|\*\s*\(?" + ARRAYS + r"\s*\+|(?<![\w.>])" + ARRAYS + r"\[[^\]]*(?:idx|qc|mo|state_at)", s)
        cast = re.search(r"static_cast<(?:const )?T \*>\([^()]*\)\s*\[", s)
        if (wide or element or cast) and "FPK_IN" not in s and "constexpr" not in s:
            bare.append(s)
    assert not bare, bare
