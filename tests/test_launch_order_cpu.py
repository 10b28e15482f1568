"""What a programmatic dependent launch may read before it waits.

Such a kernel can start before the grid ahead of it has finished, so that
everything it reads before ``pdl_wait`` has to be complete by other means: its
parameters, and the twiddle table, which ``dos_create`` builds and synchronises
on before the first such launch.  Read from the sources: a missing wait shows
neither on a CPU nor, by timing alone, on a GPU."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2604_02624_gb300", "csrc")
FILES = ("dos_pass.cuh", "dos_pass_bulk.cuh", "dos_loss.cu", "dos_setup.cu", "dos_gemm.cu")


def _code(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", text)


def test_create_finishes_the_twiddles_before_the_first_dependent_launch():
    src = _code("dos_abi.cu")
    body = src[src.index("int build(dos_ctx* x"):]
    made = body.index("launch_twiddles(")
    first = min(body.index(call, made) for call in ("ops->col(", "ops->row_back(", "choose_path("))
    assert "cudaStreamSynchronize(x->stream)" in body[made:first]


def test_nothing_but_parameters_and_twiddles_is_read_before_the_wait():
    seen = 0
    for name in FILES:
        src = _code(name)
        for m in re.finditer(r"\bpdl_wait\(\);", src):
            # from the opening of the enclosing device function
            start = max(src.rfind("__device__", 0, m.start()), src.rfind("__global__", 0, m.start()))
            head = src[start:m.start()]
            head = head[head.index("{") + 1:]
            # global memory is read through a.<array>[...], __ldg, __ldcg or an atomic; stages and barriers are shared
            reads = re.findall(r"\b(?:a|g)\.(\w+)\s*\[|(__ldc?g|atomic\w+)\s*\(", head)
            assert all(r in (("tw", ""),) for r in reads), (name, head[-400:])
            seen += 1
    assert seen >= 12


def test_the_root_table_is_in_place_only_when_its_kernel_is_queued():
    """A failed first use of displaced layers must not leave a table that looks
    made: the context's pointer is set after the launch that fills it."""
    src = _code("dos_abi.cu")
    assert "alloc(&c->sq," not in src
    assert 0 < src.index("launch_sqtable(") < src.index("c->sq = ")
