"""The producers of the tensor-core kernels wait for their own copies before the CTA
ends (tma_drain): which barriers and phases that is, restated on the ring's
arithmetic, and that every kernel with a producer does it."""
import os
import re

import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                   "paper_1310_6380_gb300", "csrc", "tc_gemm.cu")


@pytest.mark.parametrize("stages", [1, 2, 3, 4, 6])
@pytest.mark.parametrize("issued", range(14))
def test_covers_every_copy_in_flight(stages, issued):
    waits = [(i % stages, (i // stages) & 1) for i in range(max(0, issued - stages), issued)]
    # copy i uses slot i % stages in its phase i // stages; a slot is filled again
    # only after its copy was consumed, so at most the last of each slot is in flight
    last = {i % stages: (i // stages) & 1 for i in range(issued)}
    assert dict(waits) == last and len(waits) == len(last)


def test_every_producer_drains():
    src = open(SRC).read()
    kernels = re.split(r"__global__ void", src)[1:]
    producers = [k for k in kernels if "tma_load_3d(" in k.split("\n}\n")[0]]
    assert len(producers) == 3
    for k in producers:
        body = k.split("\n}\n")[0]
        assert body.count("tma_drain(") == 1
        assert body.rindex("tma_load_3d(") < body.index("tma_drain(") < body.index("MMA" if "MMA issuer" in body else "warp == 1")
