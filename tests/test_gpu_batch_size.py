"""Batches of very many items (needs a GB300 with 100 GB free: each item keeps 1 MB of tables)."""
import time

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    import __graft_entry__ as g
    g.build()
    from paper_2109_10375_gb300 import binding
    return binding


@pytest.mark.parametrize("items", [65_537])
def test_batch_of_more_items_than_a_grid_has_rows(B, monkeypatch, items):
    # 65535 is the most CTAs a grid takes along y and z
    from paper_2109_10375_gb300 import synth
    if torch.cuda.mem_get_info()[0] < 100e9:
        pytest.skip("needs 100 GB of free device memory")
    monkeypatch.setenv("AMBER_AUTOTUNE", "0")
    n, box = 8, 6.25
    S, m = synth.realisation(n, box, 3, device="cuda")
    h = B.history(8.0, 4.0, 3.0)
    z = torch.zeros((items, n, n, n), device="cuda")
    with B.Context(n ** 3) as ctx:
        ref = ctx.solve(S, m, box, 3.0, h)
        batch = B.Batch([ctx], [(S, m, box, 3.0, h, z[k]) for k in range(items)])
        batch.launch()
        assert ctx.sync_status() == 0
        batch.close()
    assert torch.equal(z, ref.expand_as(z))


def test_creating_a_batch_takes_time_in_proportion(B, monkeypatch):
    # four times the items: 13 times as long when each item went over all others
    from paper_2109_10375_gb300 import synth
    if torch.cuda.mem_get_info()[0] < 100e9:
        pytest.skip("needs 100 GB of free device memory")
    monkeypatch.setenv("AMBER_AUTOTUNE", "0")
    n, box = 8, 6.25
    S, m = synth.realisation(n, box, 3, device="cuda")
    h = B.history(8.0, 4.0, 3.0)
    z = torch.zeros((40_000, n, n, n), device="cuda")
    took = {}
    with B.Context(n ** 3) as ctx:
        for items in (10_000, 10_000, 40_000):
            specs = [(S, m, box, 3.0, h, z[k]) for k in range(items)]
            t = time.perf_counter()
            batch = B.Batch([ctx], specs)
            took[items] = time.perf_counter() - t
            batch.close()
    assert took[40_000] < 8.0 * took[10_000]
