"""The bench names the Poisson passes by the form that ran, not by their times: on small meshes an
empty pass measures an interval between events that is no shorter than a pass."""
import os
import sys

import pytest

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
bench = pytest.importorskip("bench")


@pytest.mark.parametrize("form,order,ng,eliminates", [
    ("tc", 2, 24, True), ("tc4", 2, 200, True), ("tc3", 2, 96, True), ("simt", 2, 24, True), ("simt", 2, 128, True),
    ("simt", 2, 129, False), ("radix", 2, 24, False), ("tc", 4, 24, False), ("simt", 6, 24, False)])
def test_passes_are_named_by_the_form(form, order, ng, eliminates):
    kw = dict(L=64.0, Np=24, Ntiles=1, Nbuf=0, Ng=ng, fda_order=order)
    assert bench.solves_x_by_elimination(kw, form) is eliminates
    kt = {"deposit": 0.01, "kick_drift": 0.01}
    kt.update({"dst_%d" % i: 0.004 for i in range(1, 7)})       # a few us each, the empty ones too
    rows = bench.kernel_roofline(kt, kw, {"sm_mhz": 2000.0}, {"hbm_gbs": 6700.0}, form,
                                 x_elimination=eliminates)[1]
    passes = [k for k in rows if k.startswith("dst_")]
    if form == "tc3":
        assert len(passes) == 3
    else:
        want = {True: 3 if form == "simt" else 5, False: 5 if form == "simt" else 6}[eliminates]
        assert len(passes) == want and any("elimination" in k for k in passes) is eliminates
