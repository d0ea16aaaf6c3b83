"""Writes step_roundings.json: traces of the lean FP32 step kernels as the compiler fused their plain expressions
(revision 9bd7f8c).  Needs that revision built on a GPU; run from its root:

    python <path of this file> OUT.json
"""
import json
import os
import sys

sys.path[:0] = [os.getcwd(), os.path.dirname(os.path.dirname(os.path.abspath(__file__)))]

from test_gpu_roundings import CONFIGS, trace_of  # noqa: E402

if __name__ == "__main__":
    with open(sys.argv[1], "w") as f:
        json.dump({name: trace_of(**c).tolist() for name, c in CONFIGS.items()}, f)
        f.write("\n")
