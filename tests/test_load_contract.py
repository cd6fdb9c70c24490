"""The pair storages' step reads its state, links and flux field by ordinary loads: a step launched
ahead of its predecessor's end runs while that one writes, and the ensemble's launch rewrites the
buffers it reads, so no load of theirs may ask for memory that is read-only while the kernel runs."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2412_14859_gb300", "csrc")


def code_of(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def test_no_read_only_loads_where_the_memory_is_rewritten():
    for name in ("pair_tile.cuh", "ensemble.cu"):
        code = code_of(name)
        assert "__ldg(" not in code and ".nc." not in code, name


def test_launched_ahead_only_with_a_wait_of_its_own():
    """Only kernels of pair_tile.cuh carry KernelRef::pdl, and each of them waits."""
    launched = {n for n in os.listdir(CSRC) if re.search(r"\.pdl\s*=\s*1", code_of(n))}
    assert launched == {"pair_tile.cuh"}
    code = code_of("pair_tile.cuh")
    kernels = re.findall(r"__global__[^{]*\b(cg_\w+)\([^{]*\{(.*?)\n\}", code, flags=re.S)
    assert {k for k, _ in kernels} == {"cg_pair_kernel", "cg_patch_kernel"}
    assert all("wait_for_previous();" in body for _, body in kernels)
