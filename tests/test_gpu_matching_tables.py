"""Abundance matching where table size and ranks per tile are at their edges, against the FP64 oracle.

The thresholds kernel gives each CTA 31 table points; the scan gallops (mass
weighting) or walks down from a box bound (linear weightings) when a tile spans
many points, as every tile of a small grid does.  Tolerances are those of the
same comparisons elsewhere: the mass weighting's bracket is an exact integer
test, so z differs by FP32 rounding of a redshift below 20 (5e-5 covers it many
times over); the linear weightings' margins are FP32, about 1e-7 of the total
weight, which moves a cell by more than 1e-3 only where h_j is nearly flat (at
most 1e-4 of the cells, none below 10^4).
"""
import numpy as np
import pytest
import torch

from oracle import amber_oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    import __graft_entry__ as g
    g.build()
    from paper_2109_10375_gb300 import binding
    return binding


@pytest.mark.parametrize("weighting", [0, 1, 2])
@pytest.mark.parametrize("n_table,n", [(30, 20_000), (31, 20_000), (32, 20_000), (62, 9_000), (63, 8_193),
                                       (2000, 33), (2000, 32_768), (6000, 8_192)])
def test_assign_table_edges_vs_oracle(B, weighting, n_table, n):
    g = np.random.default_rng(n_table + n)
    mass = g.uniform(0.01, 3.0, n).astype(np.float32)
    order = g.permutation(n).astype(np.int32)
    h = B.history(8.0, 4.0, 3.0, n_table=n_table, weighting=weighting)
    with B.Context(n) as ctx:
        z = ctx.assign_zre(torch.from_numpy(order).cuda(), torch.from_numpy(mass).cuda(), h)
        assert ctx.sync_status() == 0
    t = O.history_table(8.0, 4.0, 3.0, n_table=n_table)
    if weighting == 0:
        zo = O.assign_zre(order, mass.astype(np.float64), t)
        assert np.max(np.abs(z.cpu().numpy() - zo)) < 5e-5
    else:
        zo = O.assign_zre_weighted(order, mass.astype(np.float64), t, weighting, 8.0, 0.3)
        d = np.abs(z.cpu().numpy().astype(np.float64) - zo)
        assert np.mean(d > 1e-3) <= (0.0 if n < 10_000 else 1e-4), (np.mean(d > 1e-3), d.max())
        assert np.quantile(d, 0.999) < 5e-5, np.quantile(d, 0.999)


@pytest.mark.parametrize("weighting", [0, 1])
@pytest.mark.parametrize("n", [8_193, (1 << 22) + 1])
def test_assign_forms_agree(B, n, weighting):
    # redshifts stored in place (masses in rank order, or gathered up to 2^22
    # cells) and through the buckets (gathered above 2^22; a result that
    # overwrites the rank-order masses): the same numbers, bit for bit
    g = torch.Generator(device="cuda").manual_seed(n + weighting)
    mass = torch.rand(n, generator=g, device="cuda") * 2.9 + 0.01
    order = torch.randperm(n, generator=g, device="cuda").to(torch.int32)
    ranked = mass[order.long()].contiguous()
    h = B.history(8.0, 4.0, 3.0, weighting=weighting)
    with B.Context(n) as ctx:
        gathered = ctx.assign_zre(order, mass, h)
        placed = ctx.assign_zre_ranked(order, ranked, h, torch.empty_like(mass))
        F = torch.empty(n, dtype=torch.float64, device="cuda")
        with_F = ctx.assign_zre_ranked(order, ranked, h, torch.empty_like(mass), F=F)
        over = ctx.assign_zre_ranked(order, ranked, h, ranked)
        assert ctx.sync_status() == 0
    assert torch.equal(gathered, placed) and torch.equal(gathered, with_F) and torch.equal(gathered, over)


@pytest.mark.parametrize("n", [1, 63, 64, 65, 8_191, 8_192, 65_537, (1 << 20) + 1, (1 << 25) + 5])
@pytest.mark.parametrize("spread", [True, False])
def test_assign_buckets(B, n, spread):
    # through the buckets (the result overwrites the rank-order masses) at the
    # edges of the bucket counts (up to 64, 33 just above a power of two), with
    # neighbouring ranks in buckets far apart or all in one: against the
    # gathered form, bit for bit, and every cell written
    g = torch.Generator(device="cuda").manual_seed(n)
    mass = torch.rand(n, generator=g, device="cuda") * 2.9 + 0.01
    order = torch.randperm(n, generator=g, device="cuda") if spread else torch.arange(n, device="cuda")
    order = order.to(torch.int32)
    ranked = mass[order.long()].contiguous()
    h = B.history(8.0, 4.0, 3.0)
    with B.Context(n) as ctx:
        gathered = ctx.assign_zre(order, mass, h)
        over = ctx.assign_zre_ranked(order, ranked, h, ranked)
        assert ctx.sync_status() == 0
    assert torch.equal(gathered, over)
    assert bool(torch.isfinite(over).all())
