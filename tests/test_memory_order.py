"""Stores into another CTA's shared memory, as the kernels' source has them."""
import re
from pathlib import Path

CSRC = Path(__file__).resolve().parent.parent / "paper_2609_31975_b200" / "csrc"


def test_stores_to_another_cta_name_an_order():
    """A plain st.shared::cluster that the other CTA polls is a data race: the readers are loops that no barrier precedes."""
    found = [(f.name, m) for f in sorted(CSRC.glob("*.cu*")) for m in re.findall(r"\bst\.[\w.:]*shared::cluster[\w.:]*", f.read_text())]
    assert found
    for name, instruction in found:
        assert re.match(r"st\.(relaxed|release)\.cluster\.|st\.async\.", instruction), (name, instruction)
