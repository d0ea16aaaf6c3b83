"""What the sources of the step kernels have to keep.  The E kernels start while the H kernel drains (programmatic
dependent launch), so they read H through plain pointers.  A __restrict__ pointer to constant values would let a
compiler read it as read-only data, above the wait for the H kernel."""
import os
import re

import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2211_16665_gb300", "csrc")


def functions(text, names):
    """{name: text} of the named functions, from the name to the closing brace in column 0."""
    found = {}
    for name in names:
        at = [m.start() for m in re.finditer(r"[ )]%s\(const StepParams" % name, text)]
        assert len(at) == 1, name
        found[name] = text[at[0]:text.index("\n}", at[0])]
    return found


@pytest.mark.parametrize("unit,names", [
    ("kern_lean.cu", {"e_plane", "e_tile", "k_e_lean"}),
    ("kern_ho.cu", {"k_e_ho", "k_e_ho4"}),
    ("kern_step.cu", {"k_e"}),
    ("kern_f64.cu", {"k_e64"}),
])
def test_e_kernels_read_h_through_plain_pointers(unit, names):
    with open(os.path.join(SRC, unit)) as f:
        found = functions(f.read(), names)
    for name, text in found.items():
        assert re.search(r"\*\s*H[xyz]?\b", text), name
        assert not re.search(r"__restrict__\s+H[xyz]?\b", text), name


@pytest.mark.parametrize("unit", ["kern_lean.cu", "kern_ho.cu"])
def test_indices_across_components_have_64_bits(unit):
    """These kernels run on components of up to 2^30 entries, so an index into three of them does not fit 32 bits."""
    assert 2 * (2 ** 30 - 1) + (2 ** 30 - 1) > 2 ** 31 - 1
    with open(os.path.join(SRC, unit)) as f:
        text = f.read()
    assert not re.search(r"\(int\)\s*(p\.vol|tp\.idx)", text)
    assert not re.search(r"\bint vol\b", text)
