"""bench.py names the near-field and M2L kernels that a form's handle runs."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)


class Handle:
    p = 10

    def __init__(self, precision, tc_m2l):
        self.precision, self.tc_m2l = precision, tc_m2l

    def query(self, what):
        return {"leaf_side": 8, "n_p2p": 592956, "n_m2l": 2246440, "n_m2l_vb": 50000, "tc_p2p": 1, "tc_m2l": self.tc_m2l}[what]


@pytest.mark.parametrize("precision,tc_m2l,p2p,m2l,products", [
    ("fp32", 0, "k_p2p_tc", "k_m2l_vol", 3), ("mixed_tf32", 1, "k_p2p_tc", "k_m2l_tc", 3), ("fp64", 0, "k_p2p_oz", "k_m2l_oz", 28)])
def test_rooflines_name_the_kernels_of_the_form(precision, tc_m2l, p2p, m2l, products):
    import bench
    _, out = bench.rooflines(Handle(precision, tc_m2l), {"p2p": 0.26, "m2l": 0.3})
    assert out["p2p"]["kernel"].split()[0] == p2p and out["m2l"]["kernel"].split()[0] == m2l
    assert out["p2p"]["executed_frac"] == pytest.approx(products * out["p2p"]["frac"])
