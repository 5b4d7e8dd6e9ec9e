"""Precision of a plain mesh density at every mesh point, the lightest ones too, against 64-bit sums (needs a GB300).

Displacements are multiples of 2^-9 cells, so that FP32 positions are exact and
only weights and sums round.  A window weight takes at most 3 roundings per
axis, their product with the mass 3 more: 12 half-ulps (2^-24).  FP32 sums of N
contributions add N of them; sums in fixed point, whose unit lies at least 40
bits below the lightest particle, N / 2 units, one rounding, and one more for
each of up to 7 further blocks that reach the point: in all, for a point of mass
v, (20 + N) 2^-24 v + N 2^-41 m_min.  N is the particles nearest to the point or
one of its 26 neighbours.
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


def _displacements(n, rms):
    """Gradient of a Gaussian field: voids and caustics; multiples of 2^-9 cells."""
    d = np.fft.rfftn(np.random.default_rng(17).normal(size=(n, n, n)))
    k = np.fft.fftfreq(n, 1.0 / n)
    kx, ky, kz = np.arange(n // 2 + 1)[None, None, :], k[None, :, None], k[:, None, None]
    k2 = kx ** 2 + ky ** 2 + kz ** 2
    k2[0, 0, 0] = np.inf
    d *= k2 ** -0.625 * np.exp(-k2 / (0.5 * n) ** 2) / k2
    psi = [np.fft.irfftn(1j * q * d, s=(n, n, n), axes=(0, 1, 2)) for q in (kx, ky, kz)]
    f = rms / np.sqrt(np.mean(np.square(psi)))
    return [(np.round(p * f * 512.0) / 512.0).astype(np.float32) for p in psi]


@pytest.mark.parametrize("order", [2, 3])
@pytest.mark.parametrize("masses", ["equal", "halves", "orders"])
@pytest.mark.parametrize("n", [32, 64])
def test_plain_density_keeps_fp32_precision_at_every_point(B, n, masses, order):
    psi = _displacements(n, 2.5 if order == 2 else 4.0)
    g = np.random.default_rng(3)
    mass = None
    if masses == "halves":  # masses of one or two octaves: still the blocks' fixed point
        mass = g.uniform(0.5, 2.0, (n, n, n)).astype(np.float32)
    elif masses == "orders":  # as collapsed fractions: 12 orders
        mass = (10.0 ** g.uniform(-12, 0, (n, n, n))).astype(np.float32)
    t = [torch.from_numpy(p).cuda() for p in psi]
    with B.Context(n ** 3) as ctx:
        got = ctx.mesh_density(tuple(t), float(n), order, False,
                               mass=None if mass is None else torch.from_numpy(mass).cuda())
        assert ctx.sync_status() == 0
    got = got.double().cpu().numpy()
    p64, m64 = [p.astype(np.float64) for p in psi], None if mass is None else mass.astype(np.float64)
    ref = O.mesh_assign(p64, m64, float(n), order)
    N = O.mesh_assign(p64, None, float(n), 1)
    for axis in range(3):
        N = N + np.roll(N, 1, axis) + np.roll(N, -1, axis)
    mean, lightest = (1.0, 1.0) if mass is None else (m64.mean(), m64.min())
    tol = (20 + N) * 2.0 ** -24 * ref + N * 2.0 ** -41 * lightest / mean
    light = (ref > 1e-6) & (ref < 1e-2)
    assert light.sum() > 500
    assert np.all(np.abs(got - ref) <= tol), np.max((np.abs(got - ref) / np.maximum(tol, 1e-300))[tol > 0])


@pytest.mark.parametrize("n", [8, 32])
@pytest.mark.parametrize("order,shift", [(1, 0.0), (2, 0.0), (3, -0.5)])
def test_an_infinite_mass_stays_where_its_window_is(B, n, order, shift):
    # particles exactly on mesh points (CIC: one point of weight 1) or half way
    # (TSC: two per axis, the third's weight is 0): the mesh is normalised by an
    # infinite total, so a point with mass becomes NaN if the mass is infinite, else 0
    psi = torch.full((n, n, n), shift, device="cuda")
    mass = torch.ones(n, n, n, device="cuda")
    mass[3, 2, 5] = float("inf")
    with B.Context(n ** 3) as ctx:
        got = ctx.mesh_density((psi, psi, psi), float(n), order, False, mass=mass)
        ctx.sync_status()
    bad = torch.zeros(n, n, n, dtype=torch.bool, device="cuda")
    if order == 3:
        bad[2:4, 1:3, 4:6] = True
    else:
        bad[3, 2, 5] = True
    assert torch.equal(got.isnan(), bad)
    assert torch.all(got[~bad] == 0)
