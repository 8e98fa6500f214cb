"""The SOR launches depend on one another programmatically, so every CTA must
wait for the launch ahead before it ends, whether it has a site of the colour or
not: read from the kernel's source, as the fault (two launches of one colour at
once) shows only for boxes whose other colour is empty, and not in their values."""
import re
from pathlib import Path

SOR = Path(__file__).resolve().parent.parent / "paper_1403_0711_gb300" / "csrc" / "sor.cu"
WAIT = 'asm volatile("griddepcontrol.wait;" ::: "memory");'


def test_no_cta_ends_before_its_wait():
    text = SOR.read_text()
    body = text[text.index("sor_kernel(double"):]
    body = body[:body.index("\n}\n")]
    body = " ".join(re.sub(r"//[^\n]*", "", body).split())
    last = body.rindex(WAIT)
    assert body.index("griddepcontrol.launch_dependents") < last
    # threads without a site may leave early, but for thread 0, which waits first
    assert body[:last].count("return;") == body[:last].count(
        f"if (threadIdx.x == 0) {WAIT} return;")
    # nothing that an earlier launch writes is read ahead of it
    assert not re.search(r"\bu\s*\[|\br\s*\[|\bo\s*\[", body[:last])
