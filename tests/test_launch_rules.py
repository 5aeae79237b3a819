"""Rules of the kernels that start while their stream's previous kernel still runs (launch() in
csrc/launch_util.cuh), read from the source: each begins by waiting for that kernel, and takes through
`const ... * __restrict__` -- the read-only path, for data that nobody writes while the kernel exists --
only tables that no kernel writes."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2207_04620_gb300", "csrc")

# host-built: prime constants, conversion and division tables, job lists, twiddles, the encoder's tables
TABLES = {
    "PrimeConst", "FoldPrime", "ConvTable", "ModDownTable", "RescaleTable", "RelinRescaleTable", "AggSrc",
    "AutomorphismJob", "ConvertJob", "KeyIpJob", "ModDownJob", "NttJob", "A::Prime", "A::Tw", "double4 roots", "int e",
}


def _dependent_kernels():
    text = "".join(open(f).read() for f in sorted(glob.glob(CSRC + "/*.cu") + glob.glob(CSRC + "/*.cuh")))
    for name in sorted(set(re.findall(r"\blaunch\(\s*(?:c\.stream|s)\s*,\s*(k_\w+)", text))):
        defs = re.findall(r"__global__[^;{]*?\b%s\s*\(([^{;]*?)\)\s*\{\s*([^;]*;)" % name, text, re.S)
        assert len(defs) == 1, name
        yield name, re.sub(r"\s+", " ", defs[0][0]), defs[0][1]


def test_dependent_kernels_wait_first():
    kernels = list(_dependent_kernels())
    assert len(kernels) > 30
    assert [n for n, _, first in kernels if first != "after_previous_kernel();"] == []


def test_dependent_kernels_read_other_kernels_words_through_plain_pointers():
    bad = []
    for name, params, _ in _dependent_kernels():
        for p in params.split(","):
            m = re.match(r"\s*const (?:typename )?([\w:]+) \*\s*__restrict__ (\w+)", p)
            if m and m.group(1) not in TABLES and "%s %s" % m.groups() not in TABLES:
                bad.append((name, p.strip()))
            assert m or "__restrict__" not in p, (name, p)
    assert bad == []
