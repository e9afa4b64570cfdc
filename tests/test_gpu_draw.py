"""The resample draw where rounding decides: chunks of the target row whose residual is nothing but a rounding error.  An id of
probability zero is never emitted, and some id always is."""
import pytest
import torch

import paper_2511_15898_b200 as G
from paper_2511_15898_b200.build import build_library

pytestmark = pytest.mark.gpu
MASK = -1.0e4


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build_library()
    G.load_library()


@pytest.mark.parametrize("first", [True, False])
def test_chunk_without_a_residual(first):
    """The whole support lies in H* and fills one chunk (its other ids masked); what fp32 sums leave of that chunk's mass is
    a rounding error.  A threshold that falls into it goes to the nearest chunk that has a residual."""
    g = torch.Generator(device="cuda").manual_seed(4)
    B, k, n = 512, 20, 3
    V = 3 * 1024
    sup = torch.arange(k, device="cuda") * 37 + (0 if first else 2048)
    q = torch.randn(B, V, generator=g, device="cuda") - 6.0
    chunk = slice(0, 1024) if first else slice(2048, 3072)
    q[:, chunk] = MASK
    p = q - 20.0
    q[:, sup] = 1.0 + torch.randn(B, k, generator=g, device="cuda")
    p[:, sup] = q[:, sup] + 0.01 * torch.randn(B, k, generator=g, device="cuda")
    s = G.solve(q, p, n, k, 1.0, 1.0)
    r = G.read_rule(s)
    assert bool((r.jstar == k).all())
    # all drafts the same token; u0 beyond its share, u1 at the end of the distribution that the chunk occupies
    toks = sup[:1].int().expand(B, n).contiguous()
    top = 1.0 - 2.0 ** -24
    uni = torch.tensor([[top, 0.0 if first else top]], device="cuda").expand(B, 2).contiguous()
    v = G.verify(s, toks, uni)
    drawn = v.accepted == 0
    assert int(drawn.sum()) > B // 2 and set(v.status.tolist()) <= {G.GR_OK, G.GR_NOT_CONVERGED}
    t = v.token[drawn]
    assert bool(((t >= 1024) if first else ((t >= 0) & (t < 2048))).all()), t.tolist()
