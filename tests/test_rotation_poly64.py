"""The polynomials of the FP64 rotation (sin and cos of f turns, |f| <= 1/8, after
the quarter turn is split off)."""
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HEADER = os.path.join(ROOT, "paper_1007_3470_gb300", "csrc", "hfs_phase.cuh")


def _constants64():
    text = open(HEADER).read()
    vals = {m.group(1): float(m.group(2))
            for m in re.finditer(r"(k(?:SinF\d+|CosF\d+|TwoPi64(?:Lo)?))\s*=\s*([-+0-9.e]+)", text)}
    return ((vals["kTwoPi64"], vals["kTwoPi64Lo"]), [vals["kSinF%d" % k] for k in range(3, 14, 2)],
            [vals["kCosF%d" % k] for k in range(2, 15, 2)])


def test_fp64_rotation_polynomials():
    """The FP64 rotation's coefficients, as stored, meet the errors stated beside
    them and are what the committed procedure gives."""
    pytest.importorskip("mpmath")
    from paper_1007_3470_gb300 import fit_rotation_poly as F
    two_pi, sc, cc = _constants64()
    es, ec = F.errors64((sc, cc))
    assert es <= 4.25e-18 and ec <= 1.35e-18
    assert (two_pi, sc, cc) == F.fit64()
