"""Operators fused into the transform passes, at the edges of their tiles, against the FP64 oracle.

n = 4 is a single-stage transform narrower than a tile; 64 and 128 are two-stage
sizes whose last tile holds one live column (the Nyquist one).  White-noise
input puts power at every Nyquist component.  FP32 transforms a few passes deep
are good to about 1e-6 of the field's scale, the products of second derivatives
to a few times that: 1e-4 of the scale, as for the other source-pipeline tests.
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


def _t(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()


def _close(got, ref, rel=1e-4):
    scale = max(np.max(np.abs(ref)), 1e-30)
    d = np.max(np.abs(got.double().cpu().numpy() - ref))
    assert d <= rel * scale, (d, scale)


@pytest.mark.parametrize("n", [4, 64, 128])
def test_lpt_and_fcoll_vs_oracle(B, n):
    d = np.random.default_rng(n).normal(scale=0.3, size=(n, n, n)).astype(np.float32)
    d64, box, D1 = d.astype(np.float64), 1.3 * n, 0.9
    D2 = -3.0 / 7.0 * D1 ** 2
    with B.Context(n ** 3) as ctx:
        psi = ctx.lpt_displacement(_t(d), box, D1, D2)
        f = {k: ctx.esf_fcoll(_t(d), box, 2.9, 0.8, 0.5, k) for k in ("sharpk", "tophat")}
        assert ctx.sync_status() == 0
    ref = O.lpt_displacement(d64, box, D1, D2)
    for a in range(3):
        _close(psi[a], ref[a])
    for k in f:
        _close(f[k], O.fcoll_esf(O.filter_field(d64, box, 2.9, k), 0.8, 0.5))


@pytest.mark.parametrize("n", [4, 32])
@pytest.mark.parametrize("order", [1, 2, 3])
def test_interlaced_density_vs_oracle(B, n, order):
    g = np.random.default_rng(10 * n + order)
    box = 1.5 * n
    # NGP particles of both meshes stay off the cell boundaries
    lo, hi = (0.05, 0.45) if order == 1 else (-1.4, 1.4)
    psi = [(g.uniform(lo, hi, (n, n, n)) * 1.5).astype(np.float32) for _ in range(3)]
    mass = g.uniform(0.2, 2.0, (n, n, n)).astype(np.float32)
    with B.Context(n ** 3) as ctx:
        got = ctx.mesh_density(tuple(_t(p) for p in psi), box, order, True, mass=_t(mass))
        assert ctx.sync_status() == 0
    p64, m64 = [p.astype(np.float64) for p in psi], mass.astype(np.float64)
    ref = O.interlace_deconvolve(O.mesh_assign(p64, m64, box, order), O.mesh_assign(p64, m64, box, order, 0.5), box,
                                 order)
    _close(got, ref)


@pytest.mark.parametrize("order", [1, 2, 3])
@pytest.mark.parametrize("kind", ["smooth", "clump", "far", "light"])
def test_density_block_forms_vs_oracle(B, order, kind):
    # a block's sums in one fixed-point word (equal masses, few particles per
    # point), in two (a clump; masses over nine decades), or straight to the
    # mesh (particles flung so far that the block's box does not fit)
    n = 32
    g = np.random.default_rng(7 * order + len(kind))
    box = 1.0 * n
    lo, hi = (0.05, 0.45) if order == 1 else (-1.4, 1.4)
    psi = g.uniform(lo, hi, (3, n, n, n))
    mass = None
    if kind == "clump":  # every particle of an 8^3 region onto one cell
        q = np.stack(np.meshgrid(*(np.arange(n),) * 3, indexing="ij")[::-1])
        inside = np.all((q >= 8) & (q < 16), axis=0)
        psi = np.where(inside, 11.2 - q, psi)
    elif kind == "far":
        psi = psi + g.integers(-n // 2, n // 2, (3, n, n, n))
    elif kind == "light":
        mass = (10.0 ** g.uniform(-9, 0, (n, n, n))).astype(np.float32)
    psi = psi.astype(np.float32)
    with B.Context(n ** 3) as ctx:
        got = ctx.mesh_density(tuple(_t(p) for p in psi), box, order, False, mass=None if mass is None else _t(mass))
        assert ctx.sync_status() == 0
    ref = O.mesh_assign(list(psi.astype(np.float64)), None if mass is None else mass.astype(np.float64), box, order)
    # FP32 positions up to 2 n cells: windows good to a few 1e-6 of a particle
    _close(got, ref, 2e-5)
    if kind == "light":  # every mesh point to FP32 accuracy, not only the heavy ones
        r = got.double().cpu().numpy()
        live = ref > 1e-7 * ref.max()
        assert np.max(np.abs(r - ref)[live] / ref[live]) < 1e-3
