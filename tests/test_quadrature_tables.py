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
