"""What the launcher picks for a row of the loss kernel, read from its source: the shape (consumer
warps, vectors a thread holds, CTAs per SM) and the cluster width by row length, for the tests that
have to reach every one of them."""

import os
import re

SOURCE = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_16798_gb300", "csrc",
                      "rl_rows.cu")


def _table(name):
    with open(SOURCE) as f:
        body = re.search(name + r"\[\] = \{(.*?)\};", f.read(), re.S).group(1)
    return [tuple(int(x) for x in t.split(",")) for t in re.findall(r"\{([-\d, ]+)\}", body)]


SHAPES = _table("kShapes")
PICKS = {"bf16": _table("kPicksBf16"), "f32": _table("kPicksF32")}  # (largest V, shape, cluster width)
SHORT_BYTES = 8192      # rows up to this: a warp per row
F32_PLAIN = 129_024     # fp32 rows up to this: 7 warps x 9 vectors at 3 CTAs per SM, slices of 30 KB


def pick(dtype, V):
    """("warp", blocks a lane holds), ("f32", cluster width) or (shape, cluster width)."""
    es = 4 if dtype == "f32" else 2
    if V * es <= SHORT_BYTES:
        return "warp", 4 if V * es <= 2048 else 8 if V * es <= 4096 else 16
    if dtype == "f32" and V <= F32_PLAIN:
        return "f32", next(C for C in range(1, 17) if -(-(-(-V // C)) // 4) * 16 <= 30 * 1024 or C == 16)
    return next((s, C) for v, s, C in PICKS[dtype] if V <= v)
