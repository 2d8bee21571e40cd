"""Rules that every kernel source keeps and that no result on one GPU can show."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2205_02491_gb300", "csrc")
SOURCES = {os.path.basename(p): re.sub(r"//[^\n]*", "", open(p).read())
           for p in sorted(glob.glob(os.path.join(CSRC, "*.cu*")) + glob.glob(os.path.join(CSRC, "*.h")))}


def test_no_copy_is_multicast():
    """Each CTA fetches its own tiles: the library also runs as one replica per rank on several GPUs."""
    for name, text in SOURCES.items():
        joined = re.sub(r'"\s*"', "", text)  # adjacent string literals
        for asm in re.findall(r"cp\.async\.bulk[^;]*", joined):
            assert "multicast" not in asm, name


def kernels():
    """(file, kernel name, body) of every __global__ function defined in the sources."""
    for name, text in SOURCES.items():
        for m in re.finditer(r"__global__", text):
            head = re.compile(r"(\w+)\(").finditer(text, m.end())
            kernel = next(h.group(1) for h in head
                          if h.group(1) not in ("__launch_bounds__", "__cluster_dims__", "__maxnreg__"))
            start = text.index("{", m.end())
            depth, i = 1, start + 1
            while depth:
                depth += {"{": 1, "}": -1}.get(text[i], 0)
                i += 1
            yield name, kernel, text[start:i]


def test_dependent_launches_wait_before_they_return():
    """A kernel launched while the one before it drains waits for it in every thread: an early return would let the
    kernel after it start before the one before has finished."""
    launched = set()
    for text in SOURCES.values():
        launched |= set(re.findall(r"launch_pdl\(\s*(\w+)", text))
        launched |= set(re.findall(r"cudaLaunchKernelEx\(&cfg, (\w+)", text))
        launched |= set(re.findall(r"\bgo\((\w+)<", text))
    launched -= {"kernel", "void"}  # inside the helpers
    bodies = {}
    for name, kernel, body in kernels():
        bodies.setdefault(kernel, []).append((name, body))
    assert len(launched) > 15 and launched <= set(bodies), launched - set(bodies)
    for kernel in sorted(launched):
        for name, body in bodies[kernel]:
            before = body.split("grid_dependency_wait();")
            assert len(before) == 2, (name, kernel)
            assert not re.search(r"\breturn\b", re.sub(r"\[[&=]?\]\([^)]*\)( ->[^{]*)? \{[^}]*\}", "", before[0])), (name, kernel)
