"""The streaming pass at the sizes where its variants meet: one CTA or a cluster of 2, 4 or 8 CTAs per row, vocabularies
around a chunk and around what a cluster size needs, rows that are not 16-byte aligned, rows in ascending order (every
part brings candidates, the list overflows).  Support and log-sum-exp against torch in fp64."""
import pytest
import torch

import paper_2511_15898_b200 as G
from paper_2511_15898_b200.build import build_library

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build_library()
    G.load_library()


@pytest.mark.parametrize("V", [1024, 1025, 2049, 16391, 32767, 32768, 65536, 131073])
@pytest.mark.parametrize("batch", [1, 14, 15, 32, 33, 74, 75, 297])
def test_support_and_log_sum_exp(V, batch):
    for dt, k, ascending in ((torch.float32, 50, False), (torch.bfloat16, 128, False), (torch.float32, 8, True)):
        g = torch.Generator(device="cuda").manual_seed(V + batch + k)
        q = (3 * torch.randn(batch, V, generator=g, device="cuda")).to(dt)
        p = (q.float() + torch.randn(batch, V, generator=g, device="cuda")).to(dt)
        if ascending:
            p = p.sort(dim=1).values.contiguous()
        s = G.solve(q, p, 2, k, 0.75, 1.0)
        r = G.read_rule(s)
        want = torch.sort(p, dim=1, descending=True, stable=True).indices[:, :k]
        assert torch.equal(torch.sort(want, dim=1).values.int().cpu(), torch.sort(r.ids[:, :k], dim=1).values), (dt, k)
        lse = torch.logsumexp(q.double() / 0.75, 1).cpu()
        assert float((lse - r.lse_target).abs().max()) < 1e-6, (dt, k)
        assert int((s.status > 1).sum()) == 0        # (1: a solve that did not converge, which is not this pass)
