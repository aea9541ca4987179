"""The FP32 surface choice where the tolerance band is not small against FP32 rounding: small solids at the default
tolerance, and ordinary ones at large tolerance scales (g4n_set_tolerance_scale takes any).  The FP64 formulas accept a
crossing up to half a band outside the solid's other surfaces; the choice has to be theirs there too."""
import ctypes
import os
import subprocess

import pytest

from test_pick_host import ROOT, SOLIDS

# size in mm, tolerance scale
CASES = [(1e-6, 1.0), (1e-5, 1.0), (1e-4, 1.0), (0.5, 1e5), (1.0, 1e6), (40.0, 1e6), (40.0, 1e7), (1500.0, 1e8)]


@pytest.fixture(scope="module")
def libs(tmp_path_factory):
    """pick_host.cpp with its tolerance (and the depth of its points in the bands) times each scale."""
    at = tmp_path_factory.mktemp("pick_band")
    with open(os.path.join(ROOT, "tests", "pick_host.cpp")) as f:
        text = f.read()
    for old, new in (("const double half = 0.5e-9;", "const double half = 0.5e-9 * TOLERANCE;"),
                     ("t += uni(-1e-9, 1e-9);", "t += uni(-1e-9, 1e-9) * TOLERANCE;")):
        assert text.count(old) == 1
        text = text.replace(old, new)
    src = str(at / "pick_band.cpp")
    with open(src, "w") as f:
        f.write(text)
    made = {}
    for tolerance in {t for _, t in CASES}:
        so = str(at / f"pick_{tolerance:g}.so")
        subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-shared", "-fPIC", f"-DTOLERANCE={tolerance!r}", "-o", so,
                        src, "-I", os.path.join(ROOT, "include"), "-I", os.path.join(ROOT, "paper_1209_5235_gb300", "csrc")],
                       check=True)
        made[tolerance] = ctypes.CDLL(so)
    return made


@pytest.mark.parametrize("size,tolerance", CASES)
@pytest.mark.parametrize("solid", SOLIDS)
def test_choice_is_the_fp64_answer_with_a_wide_band(libs, solid, size, tolerance):
    kind, seg, bore = SOLIDS[solid]
    # in its own frame; as a daughter moved by up to 2000 mm where FP64 places a solid of this size to far below the band
    for rotated in (0, 1) if size >= 0.5 else (0,):
        for mode in (0, 1):
            out, worst = (ctypes.c_longlong * 6)(), ctypes.c_double()
            libs[tolerance].pick_check(kind, seg, bore, mode, rotated, ctypes.c_double(size), ctypes.c_longlong(250000),
                                       ctypes.c_uint64(7), out, ctypes.byref(worst))
            cases, chosen, missed, unsure, wrong, out_of_range = out
            assert cases > 100 and wrong == 0 and out_of_range == 0, (rotated, mode, list(out))
