"""The exponential sums the fast solve kernel takes its quadrature nodes from (csrc/gr_quad.cuh), against 1 / x itself."""
import os
import re

import numpy as np
import pytest

HEADER = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_15898_b200", "csrc", "gr_quad.cuh")


def _tables(name, bits):
    text = open(HEADER).read()
    body = re.search(r"kSums%s\[[^\]]*\] = \{(.*?)\n\};" % bits, text, re.S)[1]
    entries = np.array([[float(a), float(b)] for a, b in re.findall(r"\{([-0-9.e+]+)f?, ([-0-9.e+]+)f?\}", body)])
    spec = text.index("struct QuadTable<%s>" % name)
    limits = [float(x) for x in re.search(r"limit\[kLevels\] = \{(.*?)\}", text[spec:])[1].replace("f", "").split(",")]
    return entries, limits


@pytest.mark.parametrize("name,bits,bound", [("double", "64", 2.01e-10), ("float", "32", 5.6e-7)])
def test_sums_reproduce_the_reciprocal(name, bits, bound):
    """Level l has 2 (l + 1) positive terms and keeps its relative error on [1, limit] (fp32: coefficients rounded to 24 bits)."""
    entries, limits = _tables(name, bits)
    assert len(entries) == len(limits) * (len(limits) + 1) and sorted(limits) == limits
    for level, limit in enumerate(limits):
        t, c = entries[level * (level + 1):(level + 1) * (level + 2)].T
        assert len(t) == 2 * (level + 1) and (np.diff(t) > 0).all() and t[0] > 0 and (c > 0).all()
        x = np.exp(np.linspace(0.0, np.log(limit), 20001))
        err = np.abs(1.0 - x * (np.exp(-np.outer(x, t)) @ c)).max()
        assert err <= bound, (level, limit, err)


@pytest.mark.parametrize("name,bits,terms,eps", [("double", "64", 2, 2e-10), ("double", "64", 4, 2e-10), ("float", "32", 4, 5e-7), ("float", "32", 6, 5e-7)])
def test_generator_makes_the_tables(name, bits, terms, eps):
    """The generator's sums and the tables': both stop within 1e-3 of the wanted error, which falls with the fifth power of log R and faster, so
    that limits, nodes and coefficients agree to a few 1e-4."""
    pytest.importorskip("mpmath")
    from paper_2511_15898_b200.quadrature import best_sum
    entries, limits = _tables(name, bits)
    level = terms // 2 - 1
    R, t, c = best_sum(terms, eps)
    t0, c0 = entries[level * (level + 1):(level + 1) * (level + 2)].T
    assert abs(np.log(R) / np.log(limits[level]) - 1) < 3e-4
    assert np.allclose(t, t0, rtol=3e-4, atol=0) and np.allclose(c, c0, rtol=3e-4, atol=0)
