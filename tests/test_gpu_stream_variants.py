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
        # (50 tokens and two drafts are a hard system in a few rows: one solve of 297 has been seen not to converge)
        assert set(s.status.tolist()) <= {G.GR_OK, G.GR_NOT_CONVERGED}, (dt, k)
        assert int((s.status != G.GR_OK).sum()) <= batch // 200, (dt, k)


@pytest.mark.parametrize("V,batch", [(65535, 148), (65536, 148), (65537, 149), (50257, 296), (50257, 298), (300, 593), (2048, 741), (7001, 741)])
def test_support_where_the_threads_per_row_change(V, batch):
    test_support_and_log_sum_exp(V, batch)


@pytest.mark.parametrize("dt", [torch.float32, torch.bfloat16])
def test_whole_rows_in_a_large_batch(dt):
    """Whole-vocabulary rows by the CTAs of a large batch and by those of a small one: the same bits."""
    g = torch.Generator(device="cuda").manual_seed(4)
    q = (3 * torch.randn(300, 5003, generator=g, device="cuda")).to(dt)
    p = (q.float() + torch.randn(300, 5003, generator=g, device="cuda")).to(dt)
    large, st = G.alpha_star(q, p, [2, 8], 0, 0.75, 1.0)
    small, _ = G.alpha_star(q[:37], p[:37], [2, 8], 0, 0.75, 1.0)
    assert int(st.max()) == 0 and torch.equal(small, large[:37])


@pytest.mark.parametrize("dt", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("V,k", [(1500, 20), (40000, 50), (100, 0), (3001, 0), (50257, 0)])
def test_masks_are_logits_and_only_nan_and_infinity_are_not(V, k, dt):
    """Any finite value is a logit: ids masked with values down to the type's lowest, many at a time and in both rows, leave
    the other ids' results as any other mask does.  One NaN or infinity in either row is reported."""
    g = torch.Generator(device="cuda").manual_seed(V)
    q = (2 * torch.randn(3, V, generator=g, device="cuda")).to(dt)
    p = (q.float() + torch.randn(3, V, generator=g, device="cuda")).to(dt)
    idx = torch.randperm(V, generator=g, device="cuda")[: V // 3]
    want = None
    for value in (-1.0e4, -1.0e30, -1.7e38, torch.finfo(dt).min):
        qm, pm = q.clone(), p.clone()
        qm[:, idx] = value
        pm[:, idx] = value
        s = G.solve(qm, pm, 3, k, 0.75, 0.75)
        a, st = G.alpha_star(qm, pm, [3], k, 0.75, 0.75)
        assert int(st.max()) == 0 and int((s.status == G.GR_BAD_LOGITS).sum()) == 0, value
        got = (s.alpha_star.clone(), a[:, 0], G.read_rule(s).lse_target)
        want = want or got
        assert torch.equal(got[2], want[2]), value
        assert all(float((x - y).abs().max()) < 1e-6 for x, y in zip(got[:2], want[:2])), (value, got, want)
    for value in (float("nan"), float("inf"), float("-inf")):
        for row in (q, p):
            for at in (0, V // 2, V - 1):
                bad = row.clone()
                bad[1, at] = value
                s = G.solve(bad if row is q else q, bad if row is p else p, 3, k, 0.75, 0.75)
                assert [x == G.GR_BAD_LOGITS for x in s.status.tolist()] == [False, True, False], (value, at)


def _median_us(call):
    for _ in range(3):
        call()
    ts = []
    for _ in range(21):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        call()
        b.record()
        b.synchronize()
        ts.append(a.elapsed_time(b) * 1e3)
    return sorted(ts)[len(ts) // 2]


@pytest.mark.parametrize("V", [129, 600, 1025, 2047, 2048, 2100, 3500, 4100])
def test_rows_with_long_candidate_lists(V):
    """Rows of up to 2048 ids go into the candidate list as a whole, and rows of a few chunks have a threshold too low to
    keep much out; the list is cut before it is ranked (many ties among them).  A row of 2048 ids takes no longer than one
    of 2049, which has a threshold from the start."""
    g = torch.Generator(device="cuda").manual_seed(V)
    for k in (1, 8, 127, 128):
        for levels in (3, 40, 100000):
            p = torch.randint(0, levels, (5, V), generator=g, device="cuda").float() / 7 - 3
            q = torch.randn(5, V, generator=g, device="cuda")
            r = G.read_rule(G.solve(q, p, 1, k, 1.0, 1.0))
            want = torch.sort(p, dim=1, descending=True, stable=True).indices[:, :k]
            assert torch.equal(torch.sort(want, dim=1).values.int().cpu(), torch.sort(r.ids[:, :k], dim=1).values), (k, levels)
    if V == 2048:
        x = torch.randn(300, 2 * V, generator=g, device="cuda")
        us = [_median_us(lambda a=x[:, :n].contiguous(): G.alpha_star(a, a, [2], 8, 1.0, 0.9)) for n in (V, V + 1)]
        assert us[0] < 1.25 * us[1], us


@pytest.mark.parametrize("V,batch,dt", [(128256, 300, torch.float32), (152064, 560, torch.float32), (152064, 600, torch.bfloat16),
                                        (524289, 148, torch.float32), (524289, 300, torch.float32)])
def test_wide_supports_of_long_rows_fit_the_list(V, batch, dt):
    """Random rows do not fill the candidate list, whatever the support, the vocabulary and the threads per row: a support of
    112 to 128 tokens takes about what one of 64 does (1.1 times as long; the exact selection that an overfull list leads to
    takes three times as long and more), and it is the right one."""
    g = torch.Generator(device="cuda").manual_seed(V + batch)
    q = (3 * torch.randn(batch, V, generator=g, device="cuda")).to(dt)
    p = (q.float() + torch.randn(batch, V, generator=g, device="cuda")).to(dt)
    us = {k: _median_us(lambda: G.alpha_star(q, p, [8], k, 0.7, 1.0)) for k in (64, 112, 120, 128)}
    assert max(us.values()) < 1.5 * us[64], us
    rows = slice(batch - 8, batch)
    ids = G.read_rule(G.solve(q, p, 2, 128, 0.7, 1.0)).ids[rows, :128]
    want = torch.sort(p[rows], dim=1, descending=True, stable=True).indices[:, :128]
    assert torch.equal(torch.sort(want, dim=1).values.int().cpu(), torch.sort(ids, dim=1).values)


@pytest.mark.parametrize("dt", [torch.float32, torch.bfloat16])
def test_short_rows_are_cut_before_they_are_ranked(dt):
    """Rows of up to about 1000 ids are listed whole in few vectors: the list is cut by parts of a vector (many ties among the
    elements, odd lengths), and the row takes no longer than one of 1100, whose list is cut by vectors."""
    g = torch.Generator(device="cuda").manual_seed(12)
    for V in (129, 256, 257, 263, 300, 511, 515, 519, 600, 1000, 1023, 1024, 1031):
        for k in (1, 8, 64, 65, 127, 128):
            for levels in (3, 40, 100000):
                p = (torch.randint(0, levels, (5, V), generator=g, device="cuda").float() / 7 - 3).to(dt)
                q = torch.randn(5, V, generator=g, device="cuda").to(dt)
                r = G.read_rule(G.solve(q, p, 1, k, 1.0, 1.0))
                want = torch.sort(p, dim=1, descending=True, stable=True).indices[:, :k]
                assert torch.equal(torch.sort(want, dim=1).values.int().cpu(), torch.sort(r.ids[:, :k], dim=1).values), (V, k, levels)
    x = torch.randn(400, 1100, generator=g, device="cuda").to(dt)
    us = {n: _median_us(lambda a=x[:, :n].contiguous(): G.alpha_star(a, a, [2], 8, 1.0, 0.9)) for n in (500, 600, 1000, 1100)}
    assert max(us.values()) < 1.25 * us[1100], us
