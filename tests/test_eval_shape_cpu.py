"""Launch shapes of the fitness kernels from the shared memory of their CTAs
(raster.cu): what the sizing rules set aside covers the compiled kernels' static
memory, and every shape they choose for an image fits."""
import os
import re

import pytest

from paper_2603_11404_gb300 import build

KB = 1024
CTA_LIMIT, SM_LIMIT = 227 * KB, 228 * KB  # static and dynamic memory of a CTA; all of an SM, with a KB per CTA
SCRATCH = (16 + 16 * 21) * 8  # composition scratch per instrument


def constant(name, file):
    return int(re.search(rf"{name} = (\d+)", open(os.path.join(build.CSRC, file)).read()).group(1))


def reserves():
    return {k: constant(k, "internal.cuh") for k in ("kEvalReserve", "kBatchReserve")}


def static_bytes():
    """Static shared memory of every fitness kernel, as the assembler reports it."""
    build.build()
    out, name = {}, None
    for line in open(os.path.join(build.BUILD, "raster.log")):
        m = re.search(r"Compiling entry function '(\w*k_eval\w*)'", line)
        name = m.group(1) if m else None if "Compiling entry" in line else name
        m = re.search(r"(\d+) bytes smem", line)
        if m and name:
            out[name] = int(m.group(1))
    return out


def test_reserves_cover_the_static_memory():
    r, st = reserves(), static_bytes()
    assert len(st) == 6
    for name, b in st.items():
        assert b + KB <= r["kBatchReserve" if "k_eval_batch" in name else "kEvalReserve"], name


LIST = 4 * constant("kBigListCap", "internal.cuh")  # deferred list
ACC = 4 * constant("kAccWords", "raster.cu")


def front(ni, cap, threads):
    return max(ni * SCRATCH, max(8, threads // 32) * cap * 40)


def rest(ni, H, Wq):
    return (H * Wq + 3) // 4 * 16 + ni * 5 * 96 + LIST + ACC


def per_sm(ni, H, Wq, threads, cap, reserve):
    return min(1024 // threads, SM_LIMIT // (front(ni, cap, threads) + rest(ni, H, Wq) + reserve))


def wide_threads(ni, H, Wq, reserve):
    return next((1024 // n for n in (4, 2, 1) if per_sm(ni, H, Wq, 1024 // n, 16, reserve) == n), 256)


def queue_cap(ni, H, Wq, threads, reserve):
    cap = 32
    while cap > 16 and per_sm(ni, H, Wq, threads, cap, reserve) < per_sm(ni, H, Wq, threads, 16, reserve):
        cap -= 4
    return cap if front(ni, cap, threads) + rest(ni, H, Wq) <= CTA_LIMIT else 8


@pytest.mark.parametrize("kernel", ["k_eval", "k_eval_batch"])
@pytest.mark.parametrize("ni", [1, 2])
def test_chosen_shapes_fit(ni, kernel):
    """Every height of a 1280-pixel wide image up to the largest: the CTA fits, and
    an SM holds as many as the width of the CTA was chosen for."""
    reserve = reserves()["kBatchReserve" if kernel == "k_eval_batch" else "kEvalReserve"]
    static = max(b for n, b in static_bytes().items() if ("k_eval_batch" in n) == (kernel == "k_eval_batch"))
    for H in range(1, 1281):
        threads = wide_threads(ni, H, 40, reserve)
        dyn = front(ni, queue_cap(ni, H, 40, threads, reserve), threads) + rest(ni, H, 40)
        assert static + dyn <= CTA_LIMIT, (H, threads)
        n = 1024 // threads if threads > 256 else 1
        assert n * (static + dyn + KB) <= SM_LIMIT, (H, threads)
