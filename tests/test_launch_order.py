"""What the chained kernels may do before their launch dependency resolves, read from their source.

A kernel of the chain may start before the kernel ahead of it has finished, so
what it writes or reads ahead of grid_dependency_wait is part of its
correctness, and a run shows a mistake there only when the timing is unlucky.
"""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1909_13412_gb300", "csrc")


def source(name):
    """The file without its comments."""
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", text, flags=re.S))


def block(text, at):
    """The braced block that opens at or after position `at`."""
    i = text.index("{", at)
    depth = 0
    for j in range(i, len(text)):
        depth += {"{": 1, "}": -1}.get(text[j], 0)
        if depth == 0:
            return text[i:j + 1]
    raise AssertionError("unbalanced braces")


def kernel(name, file):
    text = source(file)
    m = re.search(r"__global__[^;{]*?\b" + name + r"\(", text)
    # past the parameter list
    return block(text, text.index(")", text.index(name + "(", m.start())))


@pytest.mark.parametrize("name,file,allowed", [
    # the external forces of an exchange step, whose particle kernel is never chained
    ("k_particles", "particle_kernels.cu", {"fext"}),
    ("k_adj_particles", "adjoint_kernels.cu", set())])
def test_particle_kernels_write_nothing_ahead_of_their_dependency(name, file, allowed):
    """The lattice kernel before may still be running: it reads the marks, the
    records and the accumulators that these kernels write."""
    body = kernel(name, file)
    parts = body.split("grid_dependency_wait();")
    assert len(parts) == 3  # the triggering warp's, and the others'
    ahead = parts[0] + parts[1]
    written = re.findall(r"\bA\.(\w+)\s*\[[^;=]*\]\s*[-+|]?=[^=]", ahead)
    written += re.findall(r"\*\s*A\.(\w+)\s*[-+|]?=[^=]", ahead)
    written += re.findall(r"atomic\w+\(\s*A\.(\w+)", ahead)
    assert set(written) <= allowed
    # and the same search finds the stores that come after
    after = re.findall(r"\bA\.(\w+)\s*\[[^;=]*\]\s*[-+|]?=[^=]", parts[2])
    assert "marks" in after


CUDA_INCLUDE = "/usr/local/cuda/include"


def cuda_headers():
    found = ""
    for f in ("sm_32_intrinsics.hpp", "cuda_fp16.hpp", "cuda_bf16.hpp"):
        path = os.path.join(CUDA_INCLUDE, f)
        if not os.path.exists(path):
            pytest.skip("needs the CUDA toolkit's headers")
        found += open(path).read()
    return found


def volatile_ldcg(header, ctype):
    """Whether the toolkit's __ldcg of this type is a volatile asm: a plain one may move across the wait's."""
    m = re.search(r"__ldcg\(\s*const\s+" + ctype + r"\s*\*[^)]*\)\s*\{(.*?)\}", header, flags=re.S)
    return re.search(r"\basm\s+volatile\b", m.group(1)) is not None


def test_two_byte_populations_are_loaded_as_volatile_words():
    header = cuda_headers()
    for ctype in ("float", "double", "int", "unsigned int", "unsigned short", "uint2", "long long", "unsigned long long"):
        assert volatile_ldcg(header, ctype), ctype
    if volatile_ldcg(header, "__half") and volatile_ldcg(header, "__nv_bfloat16"):
        pytest.skip("this toolkit orders the 2-byte types' loads too")
    text = source("lbp_internal.cuh")
    for store in ("StoreBF16", "StoreF16"):
        body = block(text, text.index("struct " + store))
        assert "__ldcg(" not in body, store  # of its 2-byte type: see load_word
        for fn in ("gather", "cload"):
            assert re.search(r"load_(word|last)\(", block(body, body.index(" " + fn + "("))), (store, fn)
    assert "const unsigned short *" in block(text, text.index("unsigned short load_word("))
    # the hinted loads are asm of this library
    for m in re.finditer(r"load_last\(const [^)]*\)", text):
        assert "asm volatile" in block(text, m.end()), m.group(0)


@pytest.mark.parametrize("name,file", [
    ("k_stream_collide_forced", "lbm_kernels.cu"), ("k_stream_collide_pair", "lbm_kernels.cu"),
    ("k_stream_collide_quad", "lbm_kernels.cu"), ("k_stream_collide_staged", "lbm_staged.cu"),
    ("k_adj_lattice", "adjoint_kernels.cu")])
def test_force_overflow_is_read_through_l2(name, file):
    """The accumulators are added to by atomics of other kernels of the chain, and
    an SM may still hold the line in L1 from a step before."""
    body = kernel(name, file)
    reads = re.findall(r"[^\n;]*\bfqd?\s*(?:\[|\+)[^;]*;", body)
    reads = [r for r in reads if not re.search(r"\bfqd?\s*\[[^=]*\]\s*=[^=]", r)]
    through_l2 = ("__ldcg(fq", "take_shares(fq")  # a volatile asm, and one on a pair of them
    assert reads and all(any(f in r for f in through_l2) for r in reads), reads
    helper = source("lbm_kernels.cu")
    helper = block(helper, helper.index("take_shares("))
    assert "__ldcg(at)" in helper and volatile_ldcg(cuda_headers(), "ulonglong2")


def test_exchange_asks_for_a_buffers_attributes_once():
    """Each of an exchange call's three buffers costs one driver query (about 0.2 us)."""
    text = source("lbp_api.cu")
    assert text.count("cudaPointerGetAttributes(") == 1
    body = block(text, text.index("{", text.index("lbp_status lbp_step_exchange(")))
    assert body.count("kernel_view(") == 3
