"""The failure path of the tcgen05 kernels, by reading: a launch that finds the status word set must leave as a
whole block.  (Its race, a word set while the next launch starts, cannot be staged on a GPU without a hang.)"""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2310_00810_gb300", "csrc",
                   "unet.cu")


def test_the_block_shares_one_read_of_the_status_word():
    text = re.sub(r"//[^\n]*", "", open(SRC).read())
    # by value it is read in one place, by one thread, whose answer the whole block gets
    reads = re.findall(r"[^\n]*\*reinterpret_cast<volatile unsigned\*>\(&g_umma_status\)[^\n]*", text)
    assert len(reads) == 1
    assert re.search(r"__syncthreads_or\(threadIdx\.x == 0 &&", reads[0])
    kernels = re.findall(r"__global__[^;{]*?(k_umma_\w+)\([^{]*\{(.*?)\n\}\n", text, re.S)
    assert {name for name, _ in kernels} == {"k_umma_conv", "k_umma_wgrad"}
    for name, body in kernels:
        assert body.index("if (umma_gave_up())") < body.index("tmem_alloc"), name
        assert "return" not in body[:body.index("if (umma_gave_up())")], name
