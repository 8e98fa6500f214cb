"""The SOR launches depend on one another programmatically, so no thread may
leave the kernel before it has waited for the launch ahead: read from the
kernel's source, as the fault (two launches of one colour at once) shows only
for boxes whose other colour is empty, and not in their values."""
import re
from pathlib import Path

SOR = Path(__file__).resolve().parent.parent / "paper_1403_0711_gb300" / "csrc" / "sor.cu"


def test_no_thread_leaves_before_the_wait():
    text = SOR.read_text()
    body = text[text.index("sor_kernel(double"):]
    body = body[:body.index("\n}\n")]
    body = re.sub(r"//[^\n]*", "", body)
    wait = body.index("griddepcontrol.wait")
    assert body.index("griddepcontrol.launch_dependents") < wait
    assert "return" not in body[:wait] and "return" in body[wait:]
    # nothing that an earlier launch writes is read ahead of it
    assert not re.search(r"\bu\s*\[|\br\s*\[|\bo\s*\[", body[:wait])
