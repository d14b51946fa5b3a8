"""The early exit of the soft forward's shared blocks (k_soft_fwd in soft.cu): a
warp joins its products with those the other warps have left in shared memory,
q <- q r + q + r in FP32.  A saturated product stays saturated, also an infinite
one beside a warp that has left nothing yet."""
import os
import re

import numpy as np
import pytest

from paper_2603_11404_gb300 import build

SOURCE = open(os.path.join(build.CSRC, "soft.cu")).read()


def constant(name):
    return np.float32(re.search(rf"{name} = ([0-9.e+-]+)f", SOURCE).group(1))


def start_of_part():
    """What shared memory holds before a warp has left its products."""
    v = re.search(r"part\[warp\]\[lane\] = (\w+(?:\.\w+)?);\s*__syncthreads\(\);", SOURCE).group(1)
    return constant(v) if v[0] == "k" else np.float32(v.rstrip("f"))


@pytest.mark.parametrize("q", [7e7, 1e20, 3e38, np.inf])
def test_a_saturated_product_stays_saturated(q):
    empty = start_of_part()
    for others in ([empty] * 3, [np.float32(1.0), empty, empty], [np.float32(np.inf), empty, np.float32(1e30)]):
        v = np.float32(q)
        for r in others:
            with np.errstate(all="ignore"):
                v = np.float32(np.float64(v) * np.float64(r) + np.float64(np.float32(v + r)))
        assert v >= constant("kSaturated")
