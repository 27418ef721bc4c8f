"""One case three times, each behind a 256 MiB fill that evicts L2: the command to put under a profiler (the third
launch of a kernel is the one to capture).

    python -m synthetic.profile_case cfg2 gram            # the tree scan alone, with the algorithm named
    python -m synthetic.profile_case "step b8 n64"        # all kernels of a case of perf/cases.py
    python -m synthetic.profile_case select 1024          # draft selection over that many bf16 rows

Scan alone: the operands are uploaded as recorded q, k, v (no convolution launch), q and k are normalised inside the
scan, outputs are bf16.  Launches do not overlap."""
import sys

import torch

from paper_2609_23900_b200 import binding
from synthetic import workload as W
from synthetic.device_case import DeviceCase

CASES = {
    "cfg2": W.config2,
    "cfg3": lambda: W.config3(n_layers=8),
    "cfg3x16": lambda: W.config3(n_layers=16),
    "cfg4": lambda: W.config4("random", B=8),
    "cfgP": lambda: W.config_paper(B=8),
}


def main(argv):
    cfg = argv[1] if len(argv) > 1 else "cfg2"
    arg = argv[2] if len(argv) > 2 else "auto"
    if cfg in CASES:
        ctx = binding.Context(0)
        ctx.set_scan_algo(arg)
        ctx.set_overlap(False)
        call = DeviceCase(ctx, CASES[cfg](), use_conv=False, qk_l2norm=True, out_dtype="bf16").verify
    else:
        from perf import cases
        case = dict(kind="select", R=int(arg), V=151936, dtype="bf16") if cfg == "select" else next(c for c in cases.listed() if c["name"] == cfg)
        cases._ctx().set_overlap(False)
        state = cases.prepare(case, 1)
        call = lambda: cases.run(state)
    flush = torch.empty(256 << 20, dtype=torch.uint8, device="cuda")
    for _ in range(3):
        flush.zero_()
        call()
        torch.cuda.synchronize()
    print("ok", cfg, arg)


if __name__ == "__main__":
    main(sys.argv)
