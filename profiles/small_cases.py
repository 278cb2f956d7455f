"""The small cases of the captures in this folder: two passes of one scan (or
search) through the binding, device-resident samples.

    python3 profiles/small_cases.py NAME [NAME ...]      from the repository's root
"""
import os
import sys

sys.path.insert(0, os.getcwd())

import torch  # noqa: E402

from perf import cases  # noqa: E402

S = cases._scan
CASES = {
    # ten stations, 16 streams, 1024 channels: one chunk of 782 blocks, FP32 and FP16 spectra
    "ten": S("", 10, 8, 2, 1024, 782 * 2048),
    "ten16": S("", 10, 8, 2, 1024, 782 * 2048, precision=1),
    # 64 stations, 4096 channels: 64 blocks of 2 streams in FP32, 128 blocks of 8 streams in E4M3
    "dense": S("", 64, 2, 1, 4096, 64 * 8192, fs=64e6),
    "dense8": S("", 64, 4, 2, 4096, 128 * 8192, fs=64e6, precision=2),
    # both hands of two stations: 114 partial sums
    "cross": S("", 2, 2, 2, 1024, 16384 * 2048, cross=True),
    "fringe": {"kind": "fringe", "sub": 256, "nchan": 1024, "pad_rate": 512, "pad_delay": 8192},
}

for name in sys.argv[1:]:
    state = cases.prepare(CASES[name], 7)
    for _ in range(2):
        cases.run(state)
        torch.cuda.synchronize()
    print("done", name)
    del state
