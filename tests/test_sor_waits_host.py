"""The SOR launches depend on one another programmatically.  Threads without a site
of the colour leave before they have waited for the launch ahead, so a launch must
have a thread that stays: read from the source, as the fault (two launches of one
colour at once) shows only for boxes whose other colour is empty, and not in their
values."""
import re
from pathlib import Path

SOR = Path(__file__).resolve().parent.parent / "paper_1403_0711_gb300" / "csrc" / "sor.cu"
WAIT = 'asm volatile("griddepcontrol.wait;" ::: "memory");'


def _body(text, name):
    body = text[text.index(name):]
    return " ".join(re.sub(r"//[^\n]*", "", body[:body.index("\n}\n")]).split())


def test_threads_with_a_site_wait_before_they_read():
    body = _body(SOR.read_text(), "sor_kernel(double")
    wait = body.index(WAIT)
    assert body.index("griddepcontrol.launch_dependents") < wait
    # the only way past the wait is to have no site of the colour
    assert body[:wait].count("return;") == 1
    assert "if (t >= b.Ly * b.Wh || 2 * h + par >= b.Lx) return;" in body[:wait]
    # nothing that an earlier launch writes is read ahead of it
    assert not re.search(r"\bu\s*\[|\br\s*\[|\bo\s*\[", body[:wait])


def test_no_launch_without_a_site():
    body = _body(SOR.read_text(), "cudaError_t sor_solve(")
    assert "if ((long long)b.Lx * b.Ly * b.Lz > 1) colours = 2;" in body
    assert "for (int c = 0; c < colours && e == cudaSuccess; ++c) ok(cudaLaunchKernelEx(" in body
    # sites of colour (x + y + z) & 1: colour 0 in every box, colour 1 but in 1 x 1 x 1
    for L in [(1, 1, 1), (2, 1, 1), (1, 2, 1), (1, 1, 2), (3, 3, 3), (1, 1, 5)]:
        sites = [(x + y + z) & 1 for x in range(L[0]) for y in range(L[1]) for z in range(L[2])]
        assert 0 in sites and (1 in sites) == (len(sites) > 1)
