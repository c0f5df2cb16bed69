"""The single-domain cases of bounds_cases in FP64 (which takes no face-speed step,
batch or window), against the bounds-checked library. Prints one JSON object: case
name -> [status of swe_get_info, error_cell]."""
import json
import os
import sys

import numpy as np

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))

from paper_1912_02457_gb300 import swe  # noqa: E402
from tests.bounds_cases import cases  # noqa: E402


def main():
    res = {}
    for name, wl in cases():
        d = swe.Domain(wl.astype(np.float64), "f64")
        d.step(7)
        i = d.info(check=False)
        res[name] = [int(swe.load().swe_get_info(d.h, swe.C.byref(i))), int(i.error_cell)]
        d.close()
    print(json.dumps(res))


if __name__ == "__main__":
    main()
