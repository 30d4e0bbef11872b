"""Read-only loads (__ldg) of the kernels: only of tables that stay as they are
while a run steps.  A kernel of the step may be resident while the one before
it still writes (programmatic dependent launch), and a read-only load promises
that nobody writes the data for as long as the kernel runs."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2601_19505_gb300", "csrc")
# written when a run is created (k_tables, a copy) or between steps by a kernel
# that starts nothing early (k_factors: the coefficients)
CONSTANT = ("p.hop_tab", "p.hop32_tab", "pm.sqrt_tab", "p.eps_tab", "r_coef")


def test_readonly_loads_are_of_constant_tables():
    seen = set()
    for path in sorted(glob.glob(os.path.join(CSRC, "*"))):
        with open(path) as f:
            code = re.sub(r"//[^\n]*", "", f.read())
        assert not re.search(r"ld\.global\.nc", code), path
        for m in re.finditer(r"__ld(?:g|cv|lu)\(\s*([\w.>-]+)?", code):
            assert m.group(1) in CONSTANT, "%s: %s" % (os.path.basename(path), code[m.start():m.start() + 60])
            seen.add(m.group(1))
    assert seen == set(CONSTANT)
