"""Ranking by splitting (and the digit passes it falls back to): the one stable descending order, bit for bit.

Counts sit at the edges of its forms: one bucket, bucket regions apart from the
sort arrays (below 2^18 cells), one split (up to 1024 buckets of 3840 cells), two
splits.  Distributions: balanced ones; ties spread over the cells and ties that
lie together; both signs with a wide range of exponents.  The last two outgrow a
bucket's region at some counts and take the fallback.
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    import __graft_entry__ as g
    g.build()
    from paper_2109_10375_gb300 import binding
    return binding


def _field(kind, n):
    g = torch.Generator(device="cuda").manual_seed(n % 1000 + len(kind))
    x = torch.randn(n, generator=g, device="cuda")
    if kind == "octaves":
        return torch.exp(0.8 * x)
    if kind == "narrow":
        return 1.0 + 0.001 * x
    if kind == "equal":
        return torch.full((n,), 2.5, device="cuda")
    if kind == "ties":
        return torch.exp(0.8 * x).mul_(64.0).round_().div_(64.0)
    if kind == "lump":  # a quarter of the cells, together, share one value
        x[n // 4:n // 2] = 0.5
        return x.exp_()
    if kind == "small_lump":  # as many cells as overflow a final bucket but no first one
        x[n // 4:n // 4 + min(n // 8, 6000)] = 0.5
        return x.exp_()
    x[::7] = 0.0
    x[3::11] = -0.0
    if n > 2:
        x[1], x[2] = float("inf"), float("-inf")
    return x


@pytest.mark.parametrize("kind", ["octaves", "narrow", "equal", "ties", "lump", "small_lump", "signed"])
@pytest.mark.parametrize("n", [1, 2, 319, 321, 4096, 4609, 100_003, (1 << 18) - 1, 1 << 18, 3_932_160, 3_932_161,
                               6_000_011])
def test_rank_is_the_stable_order(B, kind, n):
    J = _field(kind, n)
    with B.Context(n) as ctx:
        a = ctx.rank(J)
        b = ctx.rank(J)  # the state a ranking leaves behind
        view = torch.cat([J.new_zeros(1), J])[1:]  # 4 bytes past an aligned address
        c = ctx.rank(view)
        assert ctx.sync_status() == 0
    ref = torch.sort(-(J + 0.0), stable=True).indices.to(torch.int32)
    assert torch.equal(a, ref) and torch.equal(b, ref) and torch.equal(c, ref)


@pytest.mark.parametrize("n", [8, 16, 32, 64, 128, 256])
@pytest.mark.parametrize("source", ["recipe", "noise"])
@pytest.mark.parametrize("weighting", [0, 1])
def test_solve_agrees_with_digit_passes(B, n, source, weighting):
    # noise: intensities of both signs, whose extremes overflow a final bucket
    # from some size on; the intensities (and the host form's masses) are then
    # put back for the digit passes
    from paper_2109_10375_gb300 import synth
    box, l = 100.0 * n / 128, 3.0
    S, m = synth.realisation(n, box, 7, device="cuda")
    if source == "noise":
        S = torch.randn(S.shape, generator=torch.Generator(device="cuda").manual_seed(n), device="cuda")
    h = B.history(8.0, 4.0, 3.0, weighting=weighting)
    z, order, mass = [], [], []
    with B.Context(n ** 3) as ctx:
        for digits in (False, True):
            if digits:
                ctx.set_tuning(n, sort_digit_bits=8, fuse_histogram=1)
            z.append(ctx.solve(S, m, box, l, h))
            J = torch.empty_like(S)
            z.append(ctx.solve(S, m, box, l, h, J_out=J))
            o = torch.empty(n ** 3, dtype=torch.int32, device="cuda")
            mr = torch.empty(n ** 3, device="cuda")
            z.append(ctx.solve_ex(S, m, box, l, h, torch.empty_like(S), o, mr))
            order.append(o)
            mass.append(mr)
            zh = torch.empty(S.shape).pin_memory()
            ctx.solve_host(S.cpu().pin_memory(), m.cpu().pin_memory(), box, l, h, zh)
            assert ctx.sync_status() == 0
            z.append(zh.cuda())
    assert all(torch.equal(z[0], x) for x in z[1:])
    assert torch.equal(order[0], order[1]) and torch.equal(mass[0], mass[1])
    ref = torch.sort(-(J.reshape(-1) + 0.0), stable=True).indices
    assert torch.equal(order[0], ref.to(torch.int32)) and torch.equal(mass[0], m.reshape(-1)[ref])


def test_solve_in_a_captured_graph(B):
    from paper_2109_10375_gb300 import synth
    n, box = 64, 50.0
    S, m = synth.realisation(n, box, 3, device="cuda")
    h = B.history(8.0, 4.0, 3.0)
    with B.Context(n ** 3) as ctx:
        ref = ctx.solve(S, m, box, 3.0, h)
        z = torch.zeros_like(S)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            ctx.solve(S, m, box, 3.0, h, out=z)
        for _ in range(2):
            z.zero_()
            g.replay()
            torch.cuda.synchronize()
            assert torch.equal(z, ref)
        assert ctx.sync_status() == 0


@pytest.mark.parametrize("specs", [[(256, 0), (64, 1), (256, 1), (256, 0), (256, 1)],
                                   [(128, k % 2) for k in range(5)] + [(256, 0), (32, 0)],
                                   [(64, k % 2) for k in range(33)]])
def test_batch_of_split_rankings(B, monkeypatch, specs):
    # sizes with over 2^23 cells share the launches of their split rankings
    # (both weightings; an item whose extremes overflow a bucket takes the
    # fallback) beside sizes ranked by digit passes, or alone
    from paper_2109_10375_gb300 import synth
    monkeypatch.setenv("AMBER_AUTOTUNE", "0")
    items, ref = [], []
    with B.Context(max(n for n, _ in specs) ** 3) as ctx:
        for k, (n, w) in enumerate(specs):
            box = 100.0 * n / 128
            S, m = synth.realisation(n, box, k, device="cuda")
            if k == 3:
                S = torch.randn(S.shape, generator=torch.Generator(device="cuda").manual_seed(5), device="cuda")
            h = B.history(7.0 + 0.04 * k, 4.0, 3.0, weighting=w)
            ref.append(ctx.solve(S, m, box, 3.0 + k, h))
            items.append((S, m, box, 3.0 + k, h, torch.empty_like(S)))
        batch = B.Batch([ctx], items)
        for _ in range(2):
            for it in items:
                it[5].zero_()
            batch.launch()
            assert ctx.sync_status() == 0
            assert all(torch.equal(it[5], r) for it, r in zip(items, ref))
        batch.close()
