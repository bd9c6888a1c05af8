"""The serving loop's estimate of an operator's device memory: the fixed-point form of the FP64 stencil is
charged only where the library allocates it (no GPU)."""
import os
import re

import pytest

from paper_0707_0131_gb300 import serving

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_threshold_is_the_library_s():
    text = open(os.path.join(ROOT, "paper_0707_0131_gb300", "csrc", "kernels.cuh")).read()
    assert int(re.search(r"FX_MIN = (\d+);", text).group(1)) == serving.FX_MIN_PAIRS


@pytest.mark.parametrize("dims,max_rhs,prec,limbs", [((8, 8, 8, 8), 1, 64, False), ((8, 8, 8, 8), 2, 64, True),
                                                     ((4, 4, 4, 4), 16, 32, False), ((8, 8, 8, 16), 1, 32, True)])
def test_limbs_are_charged_where_they_are(dims, max_rhs, prec, limbs):
    s = serving.OpSpec(key="a", dims=dims, m_q=0.1, gauge=None, prec=prec, max_rhs=max_rhs)
    V = dims[0] * dims[1] * dims[2] * dims[3]
    wide = 192 if prec == 64 else 96
    rest = V * 4 * (144 + (0 if prec == 64 else 120)) + V * wide * (s.basis_max + s.nev + 32)
    assert s.resident_bytes() - rest == (V * 576 if limbs else 0)
    work = V * max_rhs * (3 * wide + 5 * 192 + 2 * wide + 2 * 192) + V * 384 + V * wide * (s.m + 3)
    assert s.workspace_bytes() - work == (4 * V * max_rhs if limbs else 0)
