"""Optimal acceptance of whole-vocabulary rows for several draft counts at once, where the bucket search can go wrong: row
lengths around a vector and a chunk (rows that are not 16-byte aligned), masked ids, rows of few or one ratio (crowded
buckets, rows left to the sort).  Against the same prefix scan in fp64 on a sorted row."""
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
    q[2, : V // 2] = -1.0e4                                                                      # masked ids
    out, st = G.alpha_star(q, p, ns, 0, 0.75, 1.25)
    assert st.tolist() == [0] * 6
    for j, n in enumerate(ns):
        assert float((out[:, j].double() - _alpha(q, p, n, 0.75, 1.25)).abs().max()) < 1e-6, n


@pytest.mark.parametrize("V", [129, 4096, 4097, 50257])
@pytest.mark.parametrize("dt", [torch.float32, torch.bfloat16])
def test_alpha_star_of_rows_with_few_ratios(V, dt):
    """Logits on a grid that both types represent, at one temperature: the log-ratio keys are exactly tied, sixteen values in
    one row and a single one (a range of zero) in the next.  A row of more than 4096 ids of one ratio is left to the sort,
    for every draft count of the call."""
    g = torch.Generator(device="cuda").manual_seed(V)
    q = (torch.randn(3, V, generator=g, device="cuda") * 12).round().clamp(-48, 48) / 4
    p = q + torch.randint(0, 16, (3, V), generator=g, device="cuda") / 2
    p[1] = q[1]
    q, p = q.to(dt), p.to(dt)
    keys = p.double() - q.double()
    assert [len(torch.unique(row)) for row in keys] == [16, 1, 16]
    ns = [1, 2, 8, 32]
    out, st = G.alpha_star(q, p, ns, 0, 1.0, 1.0)
    assert st.tolist() == [0] * 3
    for j, n in enumerate(ns):
        assert float((out[:, j].double() - _alpha(q, p, n, 1.0, 1.0)).abs().max()) < 1e-6, n
    words = G.solve(q, p, 8, 0, 1.0, 1.0).workspace.view(torch.int32)
    record, row = (32 + 128 * 12) // 4, 3 * (1 << (V - 1).bit_length())      # bytes / 4: one record, one row of the scratch
    if V > 4096:
        # (the sort's first key, that of a ratio of one: 2^63)
        assert words[3 * record + row:3 * record + row + 2].tolist() == [0, -2 ** 31]


@pytest.mark.parametrize("dt", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("V", [50257, 152064])
@pytest.mark.parametrize("value", [-1.0e9, -1.0e10, -1.0e30, -3.3e38])
def test_masked_ids_do_not_send_the_row_to_the_sort(V, dt, value):
    """Ids masked by one value in both rows at one temperature have the key 0: the range of the keys stays that of the other
    ids, however large the value (its rounding error is not), and the bucket search separates the row.  The first word of the
    row's scratch, behind the workspace's records, says what was left to the sort."""
    g = torch.Generator(device="cuda").manual_seed(V)
    q = (3 * torch.randn(2, V, generator=g, device="cuda")).to(dt)
    p = (q.float() + torch.randn(2, V, generator=g, device="cuda")).to(dt)
    q[:, V - 100:] = value
    p[:, V - 100:] = value
    q[:, 5] = value
    p[:, 5] = value
    s = G.solve(q, p, 8, 0, 1.0, 1.0)
    words = s.workspace.view(torch.int32)
    record, row = (32 + 128 * 12) // 4, 3 * (1 << (V - 1).bit_length())      # bytes / 4: one record, one row of the scratch
    assert [int(words[2 * record + b * row]) for b in range(2)] == [0, 0]
    assert float((s.alpha_star.double() - _alpha(q, p, 8, 1.0, 1.0)).abs().max()) < 1e-6


@pytest.mark.parametrize("dt", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("ids", [1, 20, 64, 127, 128, 129, 1365, 2049])
def test_candidates_at_the_edges_of_their_paths(ids, dt):
    """Forty ratios, far enough apart for buckets of their own, of `ids` ids each: one or a few of them are candidates, taken without
    an order up to 128, in order up to 4096 and left to the sort beyond."""
    g = torch.Generator(device="cuda").manual_seed(ids)
    V = 40 * ids + 129
    q = (torch.randn(4, V, generator=g, device="cuda") * 8).round().clamp(-32, 32) / 4
    p = q + (torch.arange(V, device="cuda") % 40) / 4
    q, p = q.to(dt), p.to(dt)
    ns = [1, 2, 8, 32]
    out, st = G.alpha_star(q, p, ns, 0, 1.0, 1.0)
    assert st.tolist() == [0] * 4
    for j, n in enumerate(ns):
        assert float((out[:, j].double() - _alpha(q, p, n, 1.0, 1.0)).abs().max()) < 1e-6, n
    s = G.solve(q, p, 8, 0, 1.0, 1.0)
    assert s.status.tolist() == [G.GR_SUPPORT_TOO_LARGE] * 4 and torch.equal(s.alpha_star, out[:, 2])
    bad = q.clone()
    bad[1, 7] = float("nan")
    s = G.solve(bad, p, 8, 0, 1.0, 1.0)
    assert s.status.tolist() == [G.GR_SUPPORT_TOO_LARGE, G.GR_BAD_LOGITS] + [G.GR_SUPPORT_TOO_LARGE] * 2
    assert bool(torch.isnan(s.alpha_star[1])) and torch.equal(s.alpha_star[2:], out[2:, 2])


def _alpha_of_large(q, p, n, tt, td):
    """The same where logits are so large that a difference of scaled logits keeps nothing of the smaller one: the ratio order by the
    logits' distances from their row's maximum."""
    q, p = ((x.double() - x.double().max(1, keepdim=True).values) / t for x, t in ((q, tt), (p, td)))
    return _alpha(q, p, n, 1.0, 1.0)


@pytest.mark.parametrize("dt", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("V", [2000, 50257])
@pytest.mark.parametrize("where", ["target", "draft", "both", "two ids"])
def test_any_finite_value_is_a_logit(V, dt, where):
    """One logit of up to the type's largest value: its distribution is a point, whatever the temperature's reciprocal rounds to."""
    g = torch.Generator(device="cuda").manual_seed(V)
    values = [1.0e6, 1.0e10, 1.0e17, 1.0e18, 1.0e20, 1.0e30, 0.99 * torch.finfo(dt).max, torch.finfo(dt).max]
    q = (3 * torch.randn(len(values), V, generator=g, device="cuda")).to(dt)
    p = (q.float() + torch.randn(len(values), V, generator=g, device="cuda")).to(dt)
    v = torch.tensor(values, dtype=torch.float64, device="cuda").to(dt)
    # (the target's point on the draft's likeliest id: an acceptance well away from one)
    at = p.argmax(1)
    rows = torch.arange(len(values), device="cuda")
    if where != "draft":
        q[rows, at] = v
    if where in ("draft", "both"):
        p[rows, at] = v
    if where == "two ids":
        p[rows, (at + 1) % V] = v
    ns = [1, 2, 8, 32]
    for tt, td in [(0.6, 0.7), (0.7, 1.0), (0.75, 1.25), (0.8, 0.75), (1.25, 0.6), (1.0, 1.0)]:
        out, st = G.alpha_star(q, p, ns, 0, tt, td)
        assert st.tolist() == [0] * len(values)
        s = G.solve(q, p, 8, 0, tt, td)
        assert torch.equal(s.alpha_star, out[:, 2])
        for j, n in enumerate(ns):
            err = (out[:, j].double() - _alpha_of_large(q, p, n, tt, td)).abs()
            assert float(err.max()) < 1e-6, (tt, td, n, err.tolist())


@pytest.mark.parametrize("dt", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("V", [2000, 50257])
@pytest.mark.parametrize("masked", ["target", "draft"])
@pytest.mark.parametrize("value", [-1.0e4, -1.0e18, -1.0e30, None])
def test_ids_masked_in_one_row_only(V, dt, masked, value):
    """Ids that one of the distributions excludes, by a value of up to the type's lowest, come first (no target mass) or last (no draft mass)
    in the ratio order: their log-ratio is far outside the other ids' range, or overflows fp32."""
    value = torch.finfo(dt).min if value is None else value
    for seed, (tt, td) in enumerate([(1.0, 1.0), (0.7, 1.0), (0.75, 1.25), (1.25, 0.6)]):
        g = torch.Generator(device="cuda").manual_seed(100 * V + seed)
        q = (3 * torch.randn(6, V, generator=g, device="cuda")).to(dt)
        p = (q.float() + torch.randn(6, V, generator=g, device="cuda")).to(dt)
        gone = torch.rand(6, V, generator=g, device="cuda") < torch.tensor([0.5, 0.5, 0.1, 0.01, 0.9, 0.001], device="cuda")[:, None]
        (q if masked == "target" else p)[gone] = value
        ns = [1, 2, 8, 32]
        out, st = G.alpha_star(q, p, ns, 0, tt, td)
        assert st.tolist() == [0] * 6
        sort = G.solve(q, p, 8, 0, tt, td, G.Options(force_robust=1)).alpha_star
        assert float((out[:, 2] - sort).abs().max()) < 1e-6
        for j, n in enumerate(ns):
            err = (out[:, j].double() - _alpha_of_large(q, p, n, tt, td)).abs()
            assert float(err.max()) < 1e-6, (tt, td, n, err.tolist())


@pytest.mark.parametrize("V", [2000, 50257])
@pytest.mark.parametrize("offset", [30.0, 1.0e3, 1.0e5, -1.0e6, 3.0e7, 1.0e9])
def test_common_offsets_and_narrow_ranges(V, offset):
    """Distributions are those of the logits without a common offset.  Rounded to fp32 beside it, the range of the ratios spans a few or
    many of fp32's steps, down to 0.001."""
    g = torch.Generator(device="cuda").manual_seed(V)
    q = 3 * torch.randn(4, V, generator=g, device="cuda")
    p = q + torch.tensor([1.0, 1.0e-3, 1.0, 0.1], device="cuda")[:, None] * torch.randn(4, V, generator=g, device="cuda")
    q, p = q + offset, p + torch.tensor([0.0, 0.0, 1.0, -1.0], device="cuda")[:, None] * offset
    for tt, td in [(1.0, 1.0), (0.7, 0.7), (0.75, 1.25)]:
        out, st = G.alpha_star(q, p, [2, 8, 32], 0, tt, td)
        assert st.tolist() == [0] * 4
        for j, n in enumerate([2, 8, 32]):
            err = (out[:, j].double() - _alpha_of_large(q, p, n, tt, td)).abs()
            assert float(err.max()) < 1e-6, (tt, td, n, err.tolist())
