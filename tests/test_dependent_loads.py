"""Source check of the kernels that start before the grid before them has finished.

A kernel launched as a programmatic dependent is already running while its source is being
written.  The read-only path (``__ldg``, ``ld.global.nc``, ``const __restrict__`` pointers) is
defined only for memory that nobody writes during the kernel, and a load that is no volatile
statement may be moved across the wait: such kernels read the state by ``load_state`` alone.
A wrong load of this kind shows in no result that could be relied on, so the sources are held to it.
"""
import pathlib
import re

import pytest

CSRC = pathlib.Path(__file__).resolve().parent.parent / "paper_1402_5487_gb300" / "csrc"
READ_ONLY = re.compile(r"__ldg|__ldcg|__ldca|ld\.global\.nc|ld\.global\.cg")
READ_ONLY_POINTER = re.compile(r"const\s[^,;()]*\*\s*__restrict__")
#: written by nobody while kernels run: a batch's table of parameters and list of pieces
TABLES = ("const PairParams* __restrict__ inst", "const FusePiece* __restrict__ pieces")


def code(name):
    text = re.sub(r"//[^\n]*", "", (CSRC / name).read_text())
    return re.sub(r"/\*.*?\*/", "", text, flags=re.S)


def functions(text):
    """(signature, body) of every function with a body at the text's outer levels."""
    for m in re.finditer(r"__(?:global|device)__[^;{}]*?\([^;{}]*\)[^;{}]*\{", text):
        depth, i = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
        yield m.group(0), text[m.end():i]


def dependent_kernels():
    out = []
    for f in sorted(CSRC.glob("*.cu*")):
        out += [(f.name, s, b) for s, b in functions(code(f.name)) if "__global__" in s and "step_wait()" in b]
    return out


def test_every_dependent_kernel_is_found():
    names = {re.search(r"(\w+)\s*\((?!.*\bbounds)", s.split("__launch_bounds__")[-1].split(")", 1)[-1]).group(1)
             for _, s, _ in dependent_kernels()}
    launched = set()
    for f in CSRC.glob("*.cu*"):
        for call in re.findall(r"launch_(?:dependent|dependent_smem|by_waves|large)\([^;]*;", code(f.name)):
            launched |= set(re.findall(r"\bk_\w+", call))
    assert len(names) >= 10 and len(launched) >= 8 and launched <= names, launched - names


@pytest.mark.parametrize("name", ["plbm_device.cuh", "plbm_pair.cuh", "plbm_fuse.cuh"])
def test_headers_of_the_step_kernels_have_no_read_only_load(name):
    assert not READ_ONLY.findall(code(name))


def test_dependent_kernels_read_the_state_by_load_state():
    for name, sig, body in dependent_kernels():
        for t in TABLES:
            sig = sig.replace(t, "")
        assert not READ_ONLY_POINTER.search(sig), (name, sig)
        assert not READ_ONLY.findall(body), (name, sig)
    # what a kernel of the 3D file passes its source to
    for sig, body in functions(code("plbm_step3.cu")):
        if "zpair_update" in sig:
            assert not READ_ONLY_POINTER.search(sig) and not READ_ONLY.findall(body)
