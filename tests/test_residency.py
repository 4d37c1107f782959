"""Blocks per SM that the kernels' launch shapes rely on, from the compiler's report
of registers and shared memory (CPU only): the exact windows of the standalone dots,
the vector kernels and the diagonal products are in shared memory, so either can be
the limit. Kernels with launch shapes of their own are in test_launch_shapes.py."""
import concurrent.futures as cf
import re
import subprocess

import pytest

from paper_2302_04180_gb300 import build as B

REGS_PER_SM, SMEM_PER_SM, SMEM_PER_BLOCK = 65536, 228 * 1024, 1024  # the last: reserved for each block


def _report(tmp, source):
    r = subprocess.run([B.nvcc(), "-Xptxas=-v", *B.ARCH, *B.NVCC_FLAGS, "-c", f"{B.CSRC}/{source}", "-o",
                        str(tmp / source.replace(".cu", ".o"))], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    out, name, spill = {}, None, 0
    for line in r.stderr.splitlines():
        m = re.search(r"Compiling entry function '(\S+)'", line)
        if m:
            name = m.group(1)
        m = re.search(r"(\d+) bytes spill stores", line)
        if m:
            spill = int(m.group(1))
        m = re.search(r"Used (\d+) registers(?:.*?(\d+) bytes smem)?", line)
        if m and name:
            out[name] = (int(m.group(1)), int(m.group(2) or 0), spill)
            name = None
    return out


@pytest.fixture(scope="module")
def report(tmp_path_factory):
    tmp = tmp_path_factory.mktemp("residency")
    out = {}
    with cf.ThreadPoolExecutor() as ex:
        for r in ex.map(lambda s: _report(tmp, s), ["kernels_solver.cu", "kernels_step.cu", "kernels_spmv.cu", "kernels_dot.cu",
                                                    "kernels_small.cu"]):
            out.update(r)
    return out


def _find(report, *parts):
    hits = [k for k in report if all(p in k for p in parts)]
    assert len(hits) == 1, (parts, hits)
    return report[hits[0]]


def _blocks(entry, threads):
    regs, smem, _ = entry
    by_regs = REGS_PER_SM // ((regs + 7) // 8 * 8 * 32 * (threads // 32))
    return min(by_regs, SMEM_PER_SM // (smem + SMEM_PER_BLOCK))


# kernel, threads, blocks per SM that its grid counts on
SHAPES = [
    (("k_cls_k4", "ExactRows"), 256, 4),
    (("k_pipe_p1", "ExactRows"), 256, 2),  # (three fit; its grid takes two)
    (("9k_pipe_p3", "ExactRows"), 256, 2),
    (("k_cls_k1", "ExactR", "Lin7E"), 256, 3),
    (("k_cls_k3", "ExactR", "Lin7E"), 256, 3),
    (("k_cls_k1", "ExactR", "Lin32E"), 128, 3),
    (("k_cls_k3", "ExactR", "Lin32E"), 128, 3),
    (("k_spmv_diagILi7E",), 256, 3),
    (("k_spmv_diagILi32E",), 128, 3),
    (("k_exdotILi16ELb0E",), 256, 3),
    (("k_step_cls_k4", "ExactRows"), 256, 4),
    (("k_step_pipe_p1", "ExactRows"), 256, 3),
    (("k_step_pipe_p3", "ExactRows"), 256, 2),
    (("k_step_diag_k1",), 256, 3),
    (("k_step_diag_k3",), 256, 3),
]


@pytest.mark.parametrize("parts,threads,blocks", SHAPES, ids=lambda v: "_".join(v) if isinstance(v, tuple) else None)
def test_blocks_per_sm(report, parts, threads, blocks):
    entry = _find(report, *parts)
    assert _blocks(entry, threads) >= blocks, (parts, entry)


def test_the_one_cluster_solve_leaves_room_for_the_system(report):
    """One block of 512 threads per SM, whose own arrays leave at least 180 KB of the
    shared memory for the matrix and the vectors."""
    for variant in ("k_smallILb0E", "k_smallILb1E"):
        regs, smem, _ = entry = _find(report, variant)
        assert _blocks(entry, 512) >= 1 and 227 * 1024 - smem >= 180 * 1000, (variant, entry)


def test_kernels_with_windows_in_shared_memory_hardly_spill(report):
    """At most a few words (the windows were moved there so that the loads in flight keep
    the registers)."""
    for parts in (("k_cls_k4", "ExactRows"), ("9k_pipe_p3", "ExactRows"), ("k_exdotILi16ELb0E",), ("k_cls_k1", "ExactR", "Lin7E"),
                  ("k_cls_k3", "ExactR", "Lin7E")):
        assert _find(report, *parts)[2] <= 16, parts
