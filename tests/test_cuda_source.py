"""Checks of the CUDA sources that no run can make: of paths that only a stopped wait takes, and of
code that a compiler may happen to make right. An .aligned instruction (the barriers, TMEM
allocations and TMEM stores among them) has to be reached by all lanes of a warp together: code that
branches on one lane before it reconverges first."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2607_14898_gb300", "csrc")


def source(name):
    return re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())


def between(src, start, end):
    at = src.index(start)
    return src[at:src.index(end, at)]


def test_cluster_barrier_and_tmem_allocations_reconverge():
    """Reached after one thread has initialised the barriers."""
    src, seen = source("fd_ptx.cuh"), set()
    for name, body in re.findall(r"__device__ __forceinline__ \w+ (\w+)\([^)]*\) \{\n(.*?)\n\}", src,
                                 flags=re.S):
        m = re.search(r"barrier\.cluster[^\"]*\.aligned|tcgen05\.alloc\.", body)
        if m:
            seen.add(name)
            assert "__syncwarp();" in body[:m.start()], name
    assert seen == {"cluster_sync", "tmem_alloc", "tmem_alloc_pair"}


def test_named_barriers_are_taken_by_converged_warps():
    """The set-up barriers of the GEMM and the attention, and the attention's turns, which follow
    the elected arrive that releases S."""
    for name in ("fd_gemm_kernel.cuh", "fd_attn.cu"):
        assert re.search(r"__syncwarp\(\);\s*if \(warp == \d\) named_barrier_arrive\(kReady", source(name))
    turn = between(source("fd_attn.cu"), "mbar_arrive(bar(kBarSFree", "take_turn(J);\n      const")
    assert re.match(r"[^\n]*\n\s*__syncwarp\(\);", turn)


def test_attention_backward_stores_to_tmem_from_converged_warps():
    """Between the elected arrive that releases S and the stores of P and dS every path reconverges
    (the wait between them is skipped for a CTA's first block)."""
    part = between(source("fd_attn_bwd.cu"), "mbar_arrive(bar(kSFree))",
                   "tmem_st_32x32b_x16(lanes + kColDs")
    assert "\n      __syncwarp();" in part


def test_chunk_counter_advances_before_any_wait_of_the_last_launch():
    """The decode's last launch advances the device's chunk counter whether or not its waits (for
    loads, MMAs, the accumulator) come to their end, as the host advances its own."""
    src = source("fd_gemm_kernel.cuh")
    body = src[src.index("gemm_kernel(const __grid_constant__"):]
    assert body.index("grid_dep_wait();") < body.index("pix.step += 1") < body.index("mbar_wait")
