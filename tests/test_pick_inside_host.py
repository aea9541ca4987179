"""DistanceToIn of a daughter from a point inside it (a query whose path names the mother): the FP32 choice gives the full FP64
formulas' answer, which for a box is zero and for the other solids the far side of the bore, if any."""
import ctypes
import os
import subprocess

import pytest

from test_pick_host import ROOT, SOLIDS


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("pick_inside") / "pick.so")
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-shared", "-fPIC", "-o", so,
                    os.path.join(ROOT, "tests", "pick_inside_host.cpp"), "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(ROOT, "paper_1209_5235_gb300", "csrc")], check=True)
    return ctypes.CDLL(so)


@pytest.mark.parametrize("scale", [0.5, 40.0, 1500.0])
@pytest.mark.parametrize("solid", SOLIDS)
def test_choice_from_inside(lib, solid, scale):
    kind, seg, bore = SOLIDS[solid]
    out = (ctypes.c_longlong * 4)()
    lib.pick_inside_check(kind, seg, bore, ctypes.c_double(scale), 0, ctypes.c_longlong(200000), ctypes.c_uint64(9), out)
    points, entered, unsure, wrong = out
    assert points > 1000 and wrong == 0, list(out)
    if solid == "box":
        assert entered == points    # zero: the point is in


@pytest.mark.parametrize("scale", [0.5, 40.0, 1500.0])
@pytest.mark.parametrize("near", [1, 2, 4])
def test_choice_where_a_box_is_left(lib, scale, near):
    """Points where the ray leaves a placed box, within 10 to 10^4 bands of the face: zero from inside, none from the band on;
    the bounds decide nearly all that lie clear of the band's edge, as the point of a track that has just left does."""
    out = (ctypes.c_longlong * 4)()
    lib.pick_inside_check(0, 0, 0, ctypes.c_double(scale), near, ctypes.c_longlong(200000), ctypes.c_uint64(10), out)
    points, entered, unsure, wrong = out
    assert points > 1000 and wrong == 0, list(out)
    assert 0 < entered < points and unsure < 1.1 * entered
