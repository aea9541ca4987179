"""The FP32 surface choice against the full FP64 formulas on the host: every chosen surface and every proved miss is the
FP64 answer, over boxes, orbs and tube segments (with and without bore, narrow and wide in phi), from points around the
solid and in its surface bands, in the solid's own frame and through an FP32 transform."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOLIDS = {"box": (0, 0, 0), "orb": (2, 0, 0), "tube": (1, 0, 0), "bored tube": (1, 0, 1), "narrow segment": (1, 1, 0),
          "narrow bored segment": (1, 1, 1), "wide segment": (1, 2, 0), "wide bored segment": (1, 2, 1)}


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("pick") / "pick.so")
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-shared", "-fPIC", "-o", so,
                    os.path.join(ROOT, "tests", "pick_host.cpp"), "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(ROOT, "paper_1209_5235_gb300", "csrc")], check=True)
    return ctypes.CDLL(so)


def check(lib, solid, mode, rotated, scale, n=60000, seed=5):
    out, worst = (ctypes.c_longlong * 6)(), ctypes.c_double()
    kind, seg, bore = SOLIDS[solid]
    lib.pick_check(kind, seg, bore, mode, rotated, ctypes.c_double(scale), ctypes.c_longlong(n),
                   ctypes.c_uint64(seed), out, ctypes.byref(worst))
    return list(out), worst.value


@pytest.mark.parametrize("scale", [0.5, 40.0, 1500.0])
@pytest.mark.parametrize("rotated", [0, 1])
@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("solid", SOLIDS)
def test_choice_is_the_fp64_answer(lib, solid, mode, rotated, scale):
    (cases, chosen, missed, unsure, wrong, out_of_range), worst = check(lib, solid, mode, rotated, scale, 300000 if mode else 60000)
    assert cases > 1000 and wrong == 0 and out_of_range == 0, (cases, chosen, missed, unsure, wrong, out_of_range)
    if solid.startswith("wide"):
        assert unsure == cases        # not convex in phi: always the full formulas
    elif mode == 0 and scale >= 40.0:
        assert unsure < 0.05 * cases  # the bounds decide nearly all


@pytest.mark.parametrize("scale", [40.0, 1500.0])
@pytest.mark.parametrize("solid", [s for s in SOLIDS if not s.startswith("wide")])
def test_rays_from_the_axis_are_decided(lib, solid, scale):
    """x . v is +0 or -0 there: the root taken does not depend on the sign of that zero."""
    (cases, chosen, missed, unsure, wrong, out_of_range), worst = check(lib, solid, 2, 0, scale)
    assert wrong == 0 and out_of_range == 0
    if "segment" not in solid:      # a segment's apex lies on the axis
        assert unsure < 0.01 * cases, (cases, chosen, missed, unsure)
