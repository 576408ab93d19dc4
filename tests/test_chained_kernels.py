"""Source rule of the chained kernels (those that begin with chain_begin()):
their grid may be resident while the kernel before still writes the data they
read, so they neither mark it __restrict__ nor load it through the read-only
path."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1904_00866_gb300", "csrc")
READ_ONLY = re.compile(r"__restrict__|__ldg|__ldcs|ld\.global\.nc|"
                       r"ld\.global\.L1::no_allocate\.nc")


def _strip(text):
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", text, flags=re.S)


def _kernels(text):
    """Each __global__ function of a source text, to its closing brace."""
    for m in re.finditer(r"__global__", text):
        depth, k = 0, text.index("{", m.start())
        for e in range(k, len(text)):
            depth += {"{": 1, "}": -1}.get(text[e], 0)
            if depth == 0:
                yield text[m.start():e + 1]
                break


def test_chained_kernels_read_plainly():
    seen = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = _strip(open(path).read())
        chained = [k for k in _kernels(text) if "chain_begin();" in k]
        seen += len(chained)
        for k in chained:
            # the first statement, before any access
            body = k[k.index("{") + 1:].lstrip()
            assert body.startswith("chain_begin();"), (path, body[:80])
            assert not READ_ONLY.search(k), (path, READ_ONLY.search(k))
        if chained and path.endswith(".cuh"):
            # and the device functions beside them, but for the shift
            # corrections, which lie in the kernel's own parameters
            rest = text.replace("const float* __restrict__ corr", "")
            assert not READ_ONLY.search(rest), path
    assert seen >= 6


def test_only_chained_kernels_are_launched_chained():
    """launch_chained takes no kernel without chain_begin()."""
    text = "".join(_strip(open(p).read())
                   for p in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))))
    chained = {re.search(r"(k_\w+)\s*\(", k).group(1)
               for k in _kernels(text) if "chain_begin();" in k}
    used = set()
    for m in re.finditer(r"launch_chained\((\w+),", text):
        name = m.group(1)
        if name == "k":   # the nearest definition above
            d = text[:m.start()].rindex("auto k = ")
            used |= set(re.findall(r"(k_\w+)<", text[d:m.start()].split(";")[0]))
        else:
            used.add(name)
    assert used and used <= chained, used - chained
