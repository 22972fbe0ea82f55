"""What a kernel does behind a wait that has expired, read from its source: it waits, with a limit of its own (mbar_drain, which the
abort flag does not cut short), for the UMMAs in flight before it frees tensor memory, and for the copies in flight into its
shared memory before it ends.  (Waits are not made to expire in the kernels themselves: test_gpu_bounded_wait.py does that in
kernels made for it.)"""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_03537_b200", "csrc")


# per file: the barriers that must be drained -- the last commit in front of the deallocation, landing loads, peers' sends
DRAINED = {
    "b2b_attention.cu": ["bar_drain", "bar_kvfull(", "bar_qfull("],
    "few_rows.cu": ["bar_acc", "bar_full(", "bar_recv", "bar_stat", "bar_max"],
    "few_rows_mlp.cu": ["bar_d2", "bar_full(", "bar_w2", "bar_recv"],
}


@pytest.mark.parametrize("name", sorted(DRAINED))
def test_copies_and_umma_in_flight_are_drained(name):
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
    drains = re.findall(r"mbar_drain\(([\w()%+ ]+)", text)
    for bar in DRAINED[name]:
        assert any(d.startswith(bar) for d in drains), (bar, drains)
    first_free = text.index("tmem_dealloc")
    assert text.index("mbar_drain(" + DRAINED[name][0]) < first_free
    if "_to_peer(" in text or "st_async" in text:     # senders stay until the receivers are done
        assert "*s_abort) tell_cluster(" in text and "*s_told)" in text and text.rindex("cluster_sync_all();") > text.rindex("mbar_drain(")


# kernels on CTA pairs, whose copies are not counted one by one: the UMMA issuers drain, and the CTA stays behind the last barrier
PAIRS = {"fused_pair.cuh": ["bar_drain"], "softmax_rows.cuh": ["bar_drain"], "b2b_gemm.cu": ["bar_drain", "bar_drain2"],
         "b2b_mlp.cu": ["bar_drain", "bar_drain + 8u"], "b2b_stream.cu": ["bar_drain"]}


@pytest.mark.parametrize("name", sorted(PAIRS))
def test_pair_kernels_drain_and_stay(name):
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
    assert re.findall(r"mbar_drain\(([^,]+),", text) == PAIRS[name]
    assert text.rindex("linger_behind_expired_wait(w)") > text.rindex("cluster_sync_all();") > text.rindex("mbar_drain(")


def test_every_kernel_with_tensor_memory_is_listed():
    with_tmem = {f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh")) and f != "sm100_primitives.cuh" and "tmem_dealloc" in open(os.path.join(CSRC, f)).read()}
    assert with_tmem == set(DRAINED) | set(PAIRS)
