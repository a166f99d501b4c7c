"""Write the bits of small solves to tests/golden/sweep_rounding.npz, for
the test that the dataflow sweep keeps the order in which it forms its sums.

The problems (tests/test_gpu_sweep_rounding.py) leave every stored fluence a
contribution from one octant only, so the order in which octants are added
does not matter and the bits are reproducible.  The stored bits are those of
the library at commit 251b4f5, whose sweep takes the rows of the moment
tables as they are: per direction, the moments at even and at odd storage
positions in two running sums that are added at the end; per moment, the
directions likewise.  Usage (on a GPU, with that library built):
    python tests/golden/make_sweep_rounding.py
"""
import os
import sys

import numpy as np

HERE = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, os.path.dirname(os.path.dirname(HERE)))

from tests import test_gpu_sweep_rounding as t  # noqa: E402


def main():
    out = {}
    for c in t.CASES:
        out[t.key(*c)], out[t.key(*c) + "_gradients"] = t.results(*c)
    np.savez_compressed(os.path.join(HERE, "sweep_rounding.npz"), **out)
    print(f"{len(out)} cases, {sum(v.size for v in out.values())} values")


if __name__ == "__main__":
    main()
