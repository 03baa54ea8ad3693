"""What a kernel launched ahead of its predecessor's end must hold to, read from the source.

A kernel passed to launch() starts while the kernel before it may still be writing.  So it waits
(follow()) before anything else, in every thread, and it takes what that kernel wrote through plain
pointers: a `const T* __restrict__` parameter of a kernel may be read by non-coherent loads, which are
defined only for memory that no one writes from the kernel's start to its end, and lets the compiler
move loads over the wait."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2402_10914_gb300", "csrc")
SOURCES = [f for f in sorted(os.listdir(CSRC)) if f.endswith(".cu")]


def source(f):
    return re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, f)).read())


def kernels(text):
    """name -> (parameter list, first statement)"""
    out = {}
    for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\([^)]*\)\s*)?(\w+)\s*\(([^{]*?)\)\s*\{\s*([^;]*;)", text):
        out[m.group(1)] = (m.group(2), m.group(3).strip())
    return out


def launched(text):
    return set(re.findall(r"\blaunch\(\s*(k\w+)", text))


def test_programmatic_launches_are_found():
    text = source("dfgks_kernels.cu")
    names = launched(text)
    assert {"k_ghosts", "k_cfl_min", "k_lines_xy", "k_lines_quad", "k_faces_xy", "k_flux_xy", "k_update", "k_lines"} <= names
    assert names <= set(kernels(text))
    # the attribute is set in one place, and no other file launches this way
    assert sum(source(f).count("ProgrammaticStreamSerialization;") for f in SOURCES) == 1


def test_they_wait_before_anything_else():
    text = source("dfgks_kernels.cu")
    ks = kernels(text)
    for name in launched(text):
        assert ks[name][1] == "follow();", name
    body = re.search(r"void follow\(\)\s*\{([^}]*)\}", text).group(1).split(";")
    assert body[0].strip() == "cudaGridDependencySynchronize()"


def test_they_read_nothing_through_non_coherent_loads():
    text = source("dfgks_kernels.cu")
    ks = kernels(text)
    for name in launched(text):
        bad = [p.strip() for p in ks[name][0].split(",") if re.search(r"const\s+\w+\s*\*\s*__restrict__", p)]
        assert not bad, (name, bad)
