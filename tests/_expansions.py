"""Whether PCM_FP64 uses the cells' expansions for a context, by the library's own thresholds."""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1505_07851_gb300", "csrc",
                   "integrals64.cu")


def on(stats, d_shells):
    txt = open(SRC).read()
    v = {k: int(n) for k, n in re.findall(r"constexpr int (F64_MP_\w+) = (\d+);", txt)}
    return stats["pairs_kept"] >= v["F64_MP_PAIRS"] and stats["M"] >= v["F64_MP_POINTS_D" if d_shells else "F64_MP_POINTS"]
