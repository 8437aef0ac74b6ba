"""Kernels that may start before their predecessor has finished: every CTA waits for it before it
leaves, read from the sources (a CTA that returns without waiting lets its grid complete early, and
the next call's kernels, ordered behind that grid alone, then run beside the predecessor)."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_28979_gb300", "csrc")


def _kernels():
    """{name: body} of every __global__ function."""
    out = {}
    for path in glob.glob(os.path.join(CSRC, "*.cu")):
        src = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__\s+void[^{;]*?\b(\w+_kernel)\s*\(", src):
            at = src.index("{", m.end())
            depth, i = 1, at + 1
            while depth:
                depth += {"{": 1, "}": -1}.get(src[i], 0)
                i += 1
            out[m.group(1)] = src[at:i]
    return out


def _overlapped():
    """Names of the kernels handed to launch_kernel and launch_kernel_clusters."""
    names = set()
    for path in glob.glob(os.path.join(CSRC, "*.cu")):
        src = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"launch_kernel(?:_clusters)?\(a\.overlap,\s*(?:KS,\s*)?(\w+)", src):
            name = m.group(1)
            if not name.endswith("_kernel"):   # a local variable
                found = re.findall(r"auto %s = ([^;]*);" % name, src)
                assert found, name
                names.update(re.findall(r"\w+_kernel", " ".join(found)))
            else:
                names.add(name)
    return names


def test_every_cta_of_an_overlapped_kernel_waits_before_it_leaves():
    kernels, overlapped = _kernels(), _overlapped()
    assert {"gate_mma_kernel", "onchip_kernel", "umma2_gemm_kernel", "simt_gemm_kernel", "replay_fmha_kernel",
            "replay_gather_kernel", "gate_kernel", "gate_tile_kernel"} <= overlapped, overlapped
    for name in overlapped:
        body = kernels[name]
        wait = body.find("pdl_enter();")
        assert wait >= 0, name
        assert not re.search(r"\breturn\b\s*;", body[:wait]), name


def test_workspaces_of_a_chain_are_not_read_through_the_non_coherent_path():
    """__ldg wants data that nothing writes while the kernel is resident; an overlapped kernel is
    resident while its predecessor writes the gate rows, the hidden rows and the selection."""
    kernels = _kernels()
    for name in _overlapped():
        for m in re.finditer(r"__ldg\(([^;]*)", kernels[name]):
            assert not re.search(r"\b(sel|grow|a2|tiles|n_tiles|rvt)\b|\.gate\b", m.group(1)), (name, m.group(0)[:80])
