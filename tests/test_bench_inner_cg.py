"""bench.py's figures for the three forms of the FP32 inner CG, which all report
as mixed_cg: bytes are counted for the kernels that ran, and no share of the
HBM bandwidth is stated for the one that keeps its vectors on chip."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)


class _Inst:
    def __init__(self, dims):
        self.dims, self.n = dims, 1
        for d in dims:
            self.n *= d


def figures(dims, first_pass):
    import bench
    inst = _Inst(dims)
    km = {"mixed_cg": (0.04, 10, 0.4), "mixed_residual64": (0.1, 1, 0.1),
          "mixed_cg_init": (0.03, 3, 0.09) if first_pass else (None, 0, 0.0)}
    res = {"kernel_ms": km}
    return inst, bench.roofline(res, inst, "c2"), bench.kernel_table(res, inst)["mixed_cg"]


@pytest.mark.parametrize("dims,first_pass,per_node", [((2048, 2048), True, 28),
                                                      ((256, 256, 256), True, 28),
                                                      ((256, 256, 256), False, 44)])
def test_streaming_forms(dims, first_pass, per_node):
    inst, r, e = figures(dims, first_pass)
    gbs = per_node * inst.n / 0.04e-3 / 1e9
    assert r["kernel"] == "mixed_cg" and r["bound"] == "hbm"
    assert r["algorithmic_bytes_per_launch"] == per_node * inst.n
    assert r["achieved"] == pytest.approx(gbs, rel=1e-3)
    assert e["achieved_gbs"] == pytest.approx(gbs, rel=1e-3)
    assert (r["traffic"] is None) == (not first_pass)


def test_resident_form_states_no_share_of_the_bandwidth():
    _, r, e = figures((2048, 2048), False)
    assert r["kernel"] == "mixed_cg" and r["bound"] == "on-chip"
    assert r["frac"] is None and r["traffic"] is None
    assert r["achieved"] == pytest.approx(40.0) and r["unit"] == "us/iteration"
    assert "achieved_gbs" not in e and "frac_of_hbm" not in e
