"""Kernels launched as programmatic dependents are resident while their predecessor writes: only
tables may go through read-only loads (__ldg, const __restrict__) in the sources they share."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1307_5824_gb300", "csrc")
# twiddles, samples, CTF tables, group ids, column table, deconvolution, K-hat, preconditioner, V, R
TABLES = {"tw", "htab", "h1", "h2", "gid", "col", "dec", "khat", "d", "V", "R"}


def read(name):
    return re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())


def test_read_only_loads_are_of_tables():
    for name in ("fft_passes.cu", "fft.cuh", "fft_planes.cuh", "spread.cu", "spread.cuh", "spread_mma.cu", "cg.cu"):
        for arg in re.findall(r"__ldg\(\s*&?\s*(?:reinterpret_cast<[^>]*>\()?\s*([A-Za-z_0-9.]+)", read(name)):
            assert arg.split(".")[-1] in TABLES, f"{name}: __ldg of {arg}"


def test_dependent_kernels_promise_nothing_about_their_buffers():
    found = 0
    for name in sorted(os.listdir(CSRC)):
        src = read(name)
        for m in re.finditer(r"__global__", src):
            head = src[m.start():src.find("{", m.start())]
            body = src[m.start():m.start() + len(head) + 400]
            if "pdl_wait();" not in body[len(head):].split("\n}\n")[0]:
                continue
            found += 1
            for arg in re.findall(r"__restrict__\s+([A-Za-z_0-9]+)", head):
                assert arg in TABLES, f"{name}: {arg} in {' '.join(head.split())[:80]}"
    assert found >= 20
