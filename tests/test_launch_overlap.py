"""Kernels whose launches overlap (launch_pdl) are resident while their
predecessors still write: only tables that no kernel of a call writes may be
read through `const __restrict__` pointers (which allow non-coherent loads), and
each kernel waits (pdl_wait) before it returns anywhere."""
import pathlib
import re

CSRC = pathlib.Path(__file__).resolve().parent.parent / "paper_2412_02413_gb300" / "csrc"
# written once, when the plan is made
TABLES = {"tw", "bins", "apod", "twx", "live", "phase", "bin_evan"}


def _sources():
    return {p.name: p.read_text() for p in sorted(CSRC.glob("*.cu"))}


def _overlapped(src):
    """Names of the kernels given to launch_pdl, directly or through a variable."""
    names = set()
    for m in re.finditer(r"launch_pdl\(p\.pdl,\s*(\w+)", src):
        if m[1].endswith("_kernel"):
            names.add(m[1])
        else:
            at = src.rindex(f"auto {m[1]} =", 0, m.start())
            names.update(re.findall(r"(\w+_kernel)\b", src[at:src.index(";", at)]))
    return names


def _kernel(src, name):
    m = re.search(r"__global__ [^;{]*?\b" + name + r"\(([^)]*)\)\s*\{", src)
    depth, i = 1, m.end()
    while depth:
        depth += {"{": 1, "}": -1}.get(src[i], 0)
        i += 1
    return m[1], src[m.end():i]


def test_overlapped_kernels_read_produced_data_coherently():
    seen = set()
    for src in _sources().values():
        for name in _overlapped(src):
            seen.add(name)
            args, body = _kernel(src, name)
            promised = set(re.findall(r"const [\w:]+ \*__restrict__ (\w+)", args))
            assert promised <= TABLES, (name, promised - TABLES)
            wait = body.index("pdl_wait()")
            assert not re.search(r"\breturn;", body[:wait]), name
    assert {"time_fft_kernel", "lateral_kernel", "prop_seg_kernel", "prop_frames_kernel", "epi_reduce_seg_kernel",
            "epi_reduce_frames_kernel", "epi_normalize_kernel"} <= seen
