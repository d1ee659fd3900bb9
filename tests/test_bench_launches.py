"""The launch counts that bench.py reports, against ncu launch lists of one evaluation (kernels alone) on a
workspace of the queried size."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402

# electrons: (n_up, n_dn, AOs)
SIZES = {158: (79, 79, 450), 434: (217, 217, 1260), 1056: (528, 528, 3040), 1731: (866, 865, 4985)}


class _Sys:
    def __init__(self, key, **tiles):
        self.n_up, self.n_dn, self.n_ao = SIZES[key]
        self.N = self.n_up + self.n_dn
        self._t = dict(gj_panel=8 if self.n_up > 640 else 16, a4_mode="tensor" if self.n_up >= 512 else "float_float",
                       c15_mode="cfree")
        self._t.update(tiles)

    def tiles(self):
        return dict(self._t)


@pytest.mark.parametrize("key,W,prec,tiles,count", [
    (1056, 37, "mixed", {}, 112), (1056, 300, "mixed", {}, 115), (1056, 600, "mixed", {}, 118),
    (1056, 2048, "mixed", {}, 131), (158, 1, "mixed", {}, 21), (158, 100, "mixed", {}, 21), (1731, 3, "mixed", {}, 286),
    (434, 601, "mixed", {}, 41), (1056, 37, "mixed", dict(c15_mode="tensor"), 110),
    (434, 64, "mixed", dict(a4_mode="fp64"), 35),
    (434, 64, "mixed", dict(a4_mode="tensor", c15_mode="float_float"), 52),
    (434, 96, "f64", {}, 32), (434, 152, "f64", {}, 4), (1056, 4, "f64", {}, 70)])
def test_counts_of_the_launch_lists(key, W, prec, tiles, count):
    assert bench.launches_per_step(_Sys(key, **tiles), prec, W, queried=True) == count
