"""The digit width and peer choices where digit passes rank whatever the field: later tomographic intervals."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    import __graft_entry__ as g
    g.build()
    from paper_2109_10375_gb300 import binding
    return binding


@pytest.mark.parametrize("n", [8, 64, 128])
def test_digit_choices_in_a_tomographic_matching(B, n):
    from paper_2109_10375_gb300 import synth
    box, l = 100.0 * n / 128, 3.0
    S0, m = synth.realisation(n, box, 0, device="cuda")
    S1, _ = synth.realisation(n, box, 1, device="cuda")
    srcs, bounds = [S0, (0.5 * S0 + 0.5 * S1).contiguous(), S1], [20.0, 8.6, 7.2, 5.0]
    h = B.history(8.0, 4.0, 3.0)
    z, passes = [], []
    with B.Context(n ** 3) as ctx:
        for bits, match in ((9, 0), (9, 1), (8, 0), (8, 1)):
            ctx.set_tuning(n, 0, bits, match)
            z.append(ctx.solve_tomographic(srcs, bounds, m, box, l, h))
            assert ctx.sync_status() == 0
            passes.append(ctx.sort_passes())
    assert all(torch.equal(z[0], x) for x in z[1:])
    assert passes[0] == passes[1] <= passes[2] == passes[3]
