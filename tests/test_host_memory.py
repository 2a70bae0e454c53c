"""What loading a model page-locks, read off the source (no GPU needed)."""
import os
import re

API = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2604_14612_b200", "csrc", "cl_api.cu")


def test_loading_needs_page_locked_memory_for_the_state_only():
    """The staging of the logits is the larger part of one page-locked block.  Where that is not to be had a model loads all the
    same, with the state alone locked, and logits are copied into the caller's memory."""
    src = re.sub(r"//[^\n]*", "", open(API).read())
    load = src[src.index('extern "C" int cl_load('):src.index("static char *ring_slot(cl_ctx *c, int l, int which) {")]
    assert re.findall(r"CU\(cudaMallocHost\(\(void \*\*\)&c->(\w+), ([^;]*)\)\);", load) == [("h_st", "sizeof(ClDevState)")]
    assert "c->h_logits" not in re.sub(r"c->h_logits = ", "", load)
    hand = src[src.index("static int hand_logits("):src.index("static int sync_state(")]
    assert "if (c->h_logits)" in hand and "cudaMemcpyDeviceToHost" in hand
