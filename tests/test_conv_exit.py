"""How the tensor-core kernels leave after a wait that ran out, read from their
source (no GPU may be made to run one out): in each of them warp 0 waits for
the copies it issued after the barrier that all warps pass, so that no warp
can fail later, and before the tensor memory goes back."""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1809_01600_gb300", "csrc",
                   "lbms_conv.cu")


def test_copies_are_drained_behind_the_last_barrier():
    text = open(SRC).read()
    kernels = re.findall(r"\n__global__ void.*?\n}\n", text, flags=re.S)
    assert len(kernels) == 3
    for k in kernels:
        assert "tma_load_2d" in k
        tail = k[k.rindex("__syncthreads();"):]
        drain, free = tail.index("if (*failed) drain_copies(full, ST, it,"), tail.index("tmem_dealloc(")
        assert drain < free and "*failed = 1" not in tail
        body = k[:k.rindex("__syncthreads();")]
        # every warp that issues says so when it gives up, and none returns past the barrier
        assert body.count("*failed = 1") == 2 and not re.search(r"\breturn\b", body)
        assert ("res_full" in k) == ("Sh::kResident ? res_full : nullptr" in tail)
