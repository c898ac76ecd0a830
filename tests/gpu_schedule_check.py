"""Child-process half of test_gpu_parity.py::test_dynamic_schedule_equals_fixed_stride:
runs the layer cases of SCHEDULE_CASES through the C ABI and saves a digest of every output
and gradient to the path given as the first argument. Run once with the default (dynamic)
tile schedule and once with MOE_GEMM_STATIC=1 (a fixed stride over the tile list), both with
MOE_GEMM_1SM=0: only the CTA pairs claim tiles, and by default most of these weight gradients
run on single SMs. The library reads both variables once per process."""
import hashlib
import json
import os
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, HERE)
sys.path.insert(0, os.path.dirname(HERE))

import torch  # noqa: E402

from gpu_helpers import case_inputs, run_gpu_layer  # noqa: E402

# T, d, E, k, F, bias: skewed loads (light and heavy groups in one list)
SCHEDULE_CASES = [
    (4000, 256, 16, 4, 512, "zipf"),
    (1500, 384, 12, 4, 640, "loguniform"),  # 128-wide column tiles
    (2500, 640, 96, 4, 384, "zipf"),  # 256-wide ones, the last one cut
    (3000, 256, 256, 8, 256, "zipf"),  # the maximum expert count
    (8192, 512, 64, 6, 512, "zipf"),
    (3000, 512, 64, 8, 512, "zipf"),  # CTA pairs with many light experts: claims of several tiles
    (5120, 2560, 10, 2, 2048, "none"),  # one claim per tile: the claim ring's second turn (see claims)
]
RING_SLOTS, PAIRS = 16, 76
NAMES = ["y", "dx", "h", "out_perm", "d_ab", "dx_perm", "dw_gate_up", "dw_down", "dw_router"]
GROUPED = {"h", "out_perm", "d_ab", "dx_perm"}  # rows past group_offsets[E] are never written


def claims(b):
    """Claims of the dW_gate_up GEMM in 256 x 256 tiles: an expert's tiles one by one from 8
    k-blocks of 128 rows on, else in units of 2, 4 or 8."""
    s, off = b.shape, b.group_offsets.tolist()
    tiles, n = (s.F // 64 + 1) // 2 * ((s.d + 255) // 256), 0
    for lo, hi in zip(off, off[1:]):
        nkb = (hi - lo) // 128
        if nkb:
            n += -(-tiles // (1 if nkb >= 8 else 2 if nkb >= 4 else 4 if nkb >= 2 else 8))
    return n


def digest(t):
    return hashlib.sha256(t.contiguous().view(torch.uint8).cpu().numpy()).hexdigest()


def run_cases():
    out = []
    for T, d, E, k, F, bias in SCHEDULE_CASES:
        b = run_gpu_layer(case_inputs(T, d, E, k, F, bias=bias, seed=T + E), E, k)
        used = int(b.group_offsets[-1])
        out.append({n: digest(getattr(b, n)[:used] if n in GROUPED else getattr(b, n)) for n in NAMES})
    # (the last case; a claim more per pair fills the ring's slots a second time)
    assert claims(b) > (RING_SLOTS + 1) * PAIRS, claims(b)
    return out


if __name__ == "__main__":
    assert os.environ.get("MOE_GEMM_1SM") == "0" and os.environ.get("MOE_GEMM_STATIC") in ("0", "1")
    with open(sys.argv[1], "w") as f:
        json.dump(run_cases(), f)
    print("schedule: saved")
