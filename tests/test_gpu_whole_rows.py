"""Optimal acceptance of whole-vocabulary rows for several draft counts at once, where the bucket search can go wrong: row
lengths around a vector and a chunk (rows that are not 16-byte aligned), crowded buckets, ties, masked ids.  Against the
same prefix scan in fp64 on a sorted row."""
import pytest
import torch

import paper_2511_15898_b200 as G
from paper_2511_15898_b200.build import build_library

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build_library()
    G.load_library()


def _alpha(q, p, n, tt, td):
    t = torch.softmax(q.double() / tt, 1)
    d = torch.softmax(p.double() / td, 1)
    order = torch.argsort(p.double() / td - q.double() / tt, dim=1, descending=True)
    psi = torch.cumsum(t.gather(1, order), 1) - torch.cumsum(d.gather(1, order), 1).clamp(max=1.0) ** n
    return 1.0 + psi.min(1).values.clamp(max=0.0)


@pytest.mark.parametrize("V", [129, 130, 1023, 1025, 4097, 50257, 152064])
@pytest.mark.parametrize("dt", [torch.float32, torch.bfloat16])
def test_alpha_star_of_whole_rows(V, dt):
    ns = [1, 2, 8, 32]
    g = torch.Generator(device="cuda").manual_seed(V)
    q = (3 * torch.randn(6, V, generator=g, device="cuda")).to(dt)
    p = (q.float() + torch.randn(6, V, generator=g, device="cuda")).to(dt)
    p[1] = (q[1].float() + torch.randint(0, 40, (V,), generator=g, device="cuda") / 2).to(dt)   # few ratio levels
    q[2, : V // 2] = -1.0e4                                                                      # masked ids
    p[3] = q[3]                                                                                  # one ratio
    out, st = G.alpha_star(q, p, ns, 0, 0.75, 1.25)
    assert st.tolist() == [0] * 6
    for j, n in enumerate(ns):
        assert float((out[:, j].double() - _alpha(q, p, n, 0.75, 1.25)).abs().max()) < 1e-6, n
