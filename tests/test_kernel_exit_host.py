"""What a GEMM kernel has in flight when one of its bounded waits gives up must land before the block leaves and its shared
memory becomes another's.  Running into that would take a kernel broken on purpose, so the sources are checked, on the CPU:
for every barrier that copies complete on, the kernel waits at its end, and no fixed delay stands in for a wait."""
import os
import re

import pytest

SOURCE = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2409_16626_b200", "csrc", "hif8_gemm.cu")
TEXT = re.sub(r"//[^\n]*", "", open(SOURCE).read())


def body(name):
    start = re.search(r"\n%s\(const __grid_constant__" % name, TEXT).end()
    return TEXT[start:TEXT.find("\n}\n", start)]


@pytest.mark.parametrize("kernel,barriers", [("hif8_gemm_narrow_kernel", ["bar_u8_full", "bar_bf_full"]),
                                             ("hif8_gemm_weights_kernel", ["bar_u8_full", "bar_bf_full"]),
                                             ("bf16_gemm_pair_kernel", ["bar_full", "bar_old"])])
def test_copies_are_waited_for(kernel, barriers):
    text = body(kernel)
    assert "tma_load" in text
    for b in barriers:
        assert f"wait_landed({b}(" in text, b


@pytest.mark.parametrize("kernel,barrier", [("hif8_gemm_narrow_kernel", "bar_bf_empty"), ("hif8_gemm_weights_kernel", "bar_bf_empty"),
                                            ("bf16_gemm_pair_kernel", "bar_empty")])
def test_mmas_are_waited_for(kernel, barrier):
    assert f"wait_landed({barrier}(" in body(kernel)


def test_every_wait_has_the_limit_and_there_is_no_fixed_delay():
    loops = re.findall(r"while \([^;{]*global_ns\(\)[^;{]*[;{]", TEXT)
    assert loops and all("kWaitLimitNs" in w for w in loops), loops


def test_last_tile_sends_no_signal_that_nobody_waits_for():
    # the MMA thread waits for the epilogue of a tile before it starts another; the arrivals of the last one would be on their way to
    # the leader, unordered by the relaxed barrier at the end, while it leaves
    text = body("hif8_gemm_weights_kernel")
    arrivals = re.findall(r"[^\n]*mbar_arrive_remote\(map_to_cta\(bar_acc_empty[^\n]*", text)
    assert len(arrivals) == 1 and "if (t + t_step < t_end && lane == 0)" in arrivals[0], arrivals
    assert "if (local > 0) ok = mbar_wait(bar_acc_empty, (local - 1) & 1" in text


def test_no_plain_store_is_under_way_to_a_cta_that_may_leave():
    # the barrier at the end is relaxed, so in a run that succeeds nothing may be stored to another CTA that this one does not wait
    # for: the count of issued tiles is read from there by who needs it, and the words that others touch are zeroed in front of the
    # block's barrier, which stands in front of the first barrier of the cluster
    text = body("hif8_gemm_weights_kernel")
    stores = [m.start() for m in re.finditer(r"st_cluster_(u32|v4)\(", text)]
    told = text.find("*abort_flag != 0", text.rfind("tc_fence_before();\n    __syncthreads();"))
    assert stores == [text.find("st_cluster_u32(", told)] and told > 0
    assert "ld_cluster_u32(map_to_cta(lay.issued(), rank ^ 1u))" in text
    setup = text[:text.find("cluster_arrive_relaxed()")]
    for word in ("gave_up", "issued"):
        assert 0 < setup.find(f"lay.{word}()) = 0") < setup.find("__syncthreads();"), word


@pytest.mark.parametrize("kernel,word", [("hif8_gemm_weights_kernel", "lay.gave_up()"), ("bf16_gemm_pair_kernel", "SmemLayout2::gave_up")])
def test_a_cta_that_gave_up_tells_the_cluster(kernel, word):
    # the others' own waits may all have succeeded while their signals to that CTA are under way: every CTA learns of it at the first
    # barrier of the end and passes a second one, with release, before it leaves
    text = body(kernel)
    end = text[text.rfind("tc_fence_before();\n    __syncthreads();"):]
    told, first = end.find("st_cluster_u32(map_to_cta("), end.find("cluster_wait()")
    first = end.find("cluster_sync_all()") if first < 0 else first
    assert 0 <= told < first and word in end[told:first]
    rest = end[first:]
    asked = rest.find(word)
    second = rest.find("cluster_sync_all()", asked)
    assert 0 <= asked < second < rest.find("tcgen05.dealloc")
    if kernel == "hif8_gemm_weights_kernel":
        assert asked < rest.find("wait_landed(bar_sums, 0, 1)") < second
