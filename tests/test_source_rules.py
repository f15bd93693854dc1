"""Rules of the CUDA sources that no run on a healthy device can show broken."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2503_01586_b200", "csrc")
# what one kernel of a search writes and a later one reads, by the names of parameters
CHAIN = ("rot", "sn", "cs", "masks", "state", "partial", "kept")


def _kernels(text):
    text = re.sub(r"/\*.*?\*/|//[^\n]*", " ", text, flags=re.S)
    out = {}
    for m in re.finditer(r"__global__\s+void\b", text):
        open_ = re.compile(r"\b(\w+)\s*\(((?:[^()]|\([^()]*\))*)\)\s*\{").search(text, m.end())
        depth, at = 1, open_.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[at], 0)
            at += 1
        out[open_.group(1)] = (open_.group(2), text[open_.end():at])
    return out


def test_chained_search_kernels_read_nothing_through_the_read_only_path():
    """The kernels of a search are dependent launches: one is resident while the one before it still writes, so that
    its inputs are not constant for the whole life of the kernel.  They must not be declared so (`const` with
    `__restrict__`: ld.global.nc, which may also move above the wait), nor read with __ldg."""
    with open(os.path.join(CSRC, "ropelite.cu")) as f:
        text = f.read()
    kernels = _kernels(text)
    assert len(kernels) >= 5 and all("ekv_pdl_wait" in body for _, body in kernels.values())
    assert "__ldg(" not in text
    bad = [(name, p.strip()) for name, (params, _) in kernels.items() for p in params.split(",")
           if "const" in p and "__restrict__" in p and re.search(r"(\w+)\s*$", p).group(1) in CHAIN]
    assert not bad
