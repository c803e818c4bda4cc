"""The exact FP16 field sums, restated on the host.

The kernels add the bits of g + 3/4 (0x3f000000 and more each, so that the third of them passes 2^31)
modulo 2^32 and take off a constant per term at the end.  Modulo 2^32 is what unsigned arithmetic
promises and signed arithmetic does not: the sources are held to unsigned accumulators, and the scheme
to the exact sums.
"""
import pathlib
import re

import numpy as np
import pytest

CSRC = pathlib.Path(__file__).resolve().parent.parent / "paper_1402_5487_gb300" / "csrc"


@pytest.mark.parametrize("name,kernel", [("plbm_aux.cu", "k_moments_f16pair"), ("plbm_step3.cu", "k_moments3_f16pair")])
def test_accumulators_are_unsigned(name, kernel):
    text = (CSRC / name).read_text()
    body = text[text.index(kernel + "("):]
    body = body[:body.index("\n}\n")]
    assert "0.75f" in body
    assert not re.search(r"\bu?int2?\b[^;]*__float_as_int|\bint2\b|\+= *__float_as_int", body)


@pytest.mark.parametrize("n", [5, 25])
@pytest.mark.parametrize("scale", [0.2498779296875, 1e-3, 2.0**-24])
def test_modular_sums_are_exact(n, scale):
    g = (np.random.default_rng(n).uniform(-1, 1, (200, n)) * scale).astype(np.float16)
    g[0], g[1] = np.float16(0.2498779296875), np.float16(-0.2498779296875)
    bits = (g.astype(np.float32) + np.float32(0.75)).view(np.uint32)
    total = np.zeros(len(g), np.uint32)
    for k in range(n):
        total += bits[:, k]
    got = (total - np.uint32(n * 0x3f400000 & 0xffffffff)).view(np.int32).astype(np.float64) * 2.0**-24
    assert np.array_equal(got, g.astype(np.float64).sum(axis=1))
