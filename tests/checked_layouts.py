"""Sweep layouts and ghost routes of larger grids run through the index-checked
build of the library (run by test_gpu_checked_layouts.py in a process with
WOMBAT_CHECKED=1), each above the 152 tiles below which a launch takes the kernel
for any layout: rings of a block and inside warps, open closed pencils, planes with
their one-zone axis, boxes with closed and outflow axes at once, passes that hold
whole rows or layers of patches and fill images along these axes only, a last pass
with fewer patches, general eps, and fields that send blocks to FP64 products.
Prints one JSON line: the check word after each scenario (0 = no out-of-range index)."""
import json
import os
import sys

import numpy as np

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

# name: (n, keywords)
GRIDS = {
    "ring_block": ((64, 40, 32), {}),
    "ring_warp": ((16, 32, 64), {}),
    "open_closed": ((48, 50, 33), {}),
    "any_layout": ((130, 32, 20), {}),
    "plane_thin": ((96, 80, 1), {}),
    "thin_x": ((1, 128, 64), {}),
    "two_zones": ((2, 96, 64), {}),
    "outflow": ((33, 30, 37), {"bc": (1, 1, 1)}),
    "mixed_closed_x": ((32, 30, 28), {"bc": (0, 1, 1)}),
    "mixed_closed_z": ((31, 30, 32), {"bc": (1, 1, 0)}),
    "plane_mixed": ((90, 70, 1), {"bc": (1, 0, 0)}),
    "rows": ((36, 36, 36), {"patches": (2, 3, 3), "batch_patches": 2}),
    "layers": ((36, 36, 36), {"patches": (3, 3, 3), "batch_patches": 9}),
    "layers_part": ((24, 24, 40), {"patches": (2, 2, 5), "batch_patches": 8}),
    "all_imaged": ((32, 32, 32), {"patches": (2, 2, 2)}),
    "rows_mixed": ((48, 24, 24), {"patches": (2, 2, 2), "batch_patches": 4, "bc": (0, 1, 0)}),
    "closed_patched": ((32, 30, 24), {"patches": (1, 3, 2), "batch_patches": 3}),
    "rings_all": ((30, 32, 34), {"patches": (2, 2, 2), "batch_patches": 1}),
    "general_eps": ((40, 33, 32), {"eps": (0.2, 0.1, 0.2, 0.05, 0.2, 0.1, 0.2), "sweby": 1.5}),
    "floors_rings": ((32, 32, 32), {"prot_rho": 1e-3, "prot_p": 1e-3}),
}


def main():
    assert os.environ.get("WOMBAT_CHECKED") == "1"
    from paper_1701_07452_gb300 import binding as wb
    from paper_1701_07452_gb300.initial_conditions import random_box
    out = {}
    wb.check_flags()  # clear
    for name, (n, kw) in GRIDS.items():
        st = random_box(n, seed=17)
        g = wb.Grid(n, length=st["length"], **kw)
        g.load_state(st)
        g.advance(2)
        g.read()
        g.divb_max()
        out[name] = wb.check_flags()
    # zones beyond the integer products' range in single blocks
    st = random_box((64, 40, 33), seed=18)
    st["W"][0, 5, 6, 7] = 2.0 ** -60
    st["W"][1, 20, 21, 22] = 2.0 ** -200
    for name, kw in (("wild_closed", {}), ("wild_outflow", {"bc": (1, 1, 1)})):
        g = wb.Grid((64, 40, 33), length=st["length"], **kw)
        g.load_state(st)
        g.advance(1)
        out[name] = wb.check_flags()
    sizes = [(64, 32, 16), (48, 50, 33), (130, 20, 12), (1, 40, 40)]
    for form in ("persistent", "staged"):
        for bc in ((0, 0, 0), (1, 0, 1)):
            bt = wb.Batch([{"n": n, "length": tuple(map(float, n)), "bc": bc} for n in sizes], work_budget=1 << 26)
            bt.set_form(form)
            for i, n in enumerate(sizes):
                bt.load_state(i, random_box(n, seed=30 + i))
            bt.set_steps(-1, 2)
            bt.advance(2)
            for i in range(len(sizes)):
                bt.read(i)
            out[f"batch_{form}_{bc[0]}"] = wb.check_flags()
    print(json.dumps(out), flush=True)


if __name__ == "__main__":
    main()
