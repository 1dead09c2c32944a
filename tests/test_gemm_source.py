"""Rules of the tensor-core product kernels (csrc/k_gemm.cu) that only a wait that gives up, or another order of the
compiler's loads, would show on a GPU: checked on the source."""
import os
import re

import pytest

SRC = open(os.path.join(os.path.dirname(__file__), "..", "paper_2512_13359_gb300", "csrc", "k_gemm.cu")).read()
KERNELS = ("k_gemm_tc", "k_gemm_rows", "k_gemm_group")


def _body(name):
    start = re.search(r"__global__[^;{]*?\b%s\(" % name, SRC).end()
    return SRC[start:SRC.index("\n}\n", start)]


@pytest.mark.parametrize("kernel", KERNELS)
def test_nothing_is_in_flight_when_a_block_leaves(kernel):
    """A producer whose wait gave up waits for the stages it has filled, and the issuer for the last of its MMAs before
    the tensor memory they write is freed."""
    b = _body(kernel)
    gave_up = b.index("if (*abort)")
    assert "wait_landed(&bar->full[" in b[gave_up:b.index("__syncwarp()", gave_up)]
    last = [m for m in re.finditer(r"mma_commit\(&bar->(\w+)", b)][-1]
    assert re.match(r"mma_commit\(&bar->(\w+)\);\s*wait_landed\(&bar->\1, [01]\);", b[last.start():])
    assert last.start() < b.index("tmem_dealloc")


@pytest.mark.parametrize("kernel", KERNELS)
def test_a_warp_gives_up_whole(kernel):
    """Tensor-memory reads are warp-wide: an epilogue warp leaves its loop, or stays, with all its lanes."""
    epilogue = re.split(r"\n  } else {\n", _body(kernel))[-1]
    assert "tmem_ld32" in epilogue
    for m in re.finditer(r"[^;]*mbar_wait\([^;]*;\s*if \(!([^;]*)\) break;", epilogue):
        assert "__all_sync" in m.group(0), m.group(0)


def test_reads_stay_behind_the_wait_for_the_previous_kernel():
    """A kernel that may start while its predecessor runs takes no operand by a read that the compiler may move ahead of
    the wait, or that may be served from a cache that the predecessor's stores bypass: addresses carry pdl_enter()'s
    zero, and no load is of the constant kind (.nc, __ldg)."""
    assert not re.search(r"(?m)^\s*pdl_enter\(\);", SRC)
    for kernel in ("k_gemm_tc", "k_gemm_rows"):
        assert re.search(r"\bint row = [^;]*\+ zero;", _body(kernel)), kernel
    tensor = SRC[:SRC.index("// fp32 on the CUDA cores.")] + SRC[SRC.index("void reduce_block("):]
    assert ".nc." not in tensor and "__ldg" not in tensor
    for name in ("reduce_block", "k_reduce"):
        head = SRC[SRC.index(name + "("):]
        assert "__restrict__ aux" not in head[:head.index("{")], name
