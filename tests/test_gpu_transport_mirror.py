"""Transport kernels on mirrored momentum cells against the oracle, bit for bit:
odd axes (cells on a mirror plane), single cells along an axis, time steps on both
sides of the drift's narrow forms, negative cells, n beyond the masses' and
the moments' narrow ranges, box sizes whose cell centres are rounded, fewer z cells
than the drift's warps."""
import numpy as np
import pytest

import oracle as O
from paper_1912_04457_gb300 import inputs as I

pytestmark = pytest.mark.gpu

CASES = [
    # nx, np, L, mask, dt (dx = 0.2), f range, force
    ((3, 4, 5), (5, 4, 7), 2.0, 0x01, 0.05, (0.0, 0.6), True),
    ((2, 1, 9), (1, 2, 3), 2.0, 0x03, 0.05, (-0.3, 0.9), True),
    ((1, 3, 2), (8, 6, 4), 0.7, 0x17, 0.1998, (-0.2, 0.9), False),     # dt/dx = 0.999
    ((4, 1, 1), (6, 7, 8), 7.3, 0x13, 0.1997, (0.0, 0.9), True),       # and just below
    ((2, 2, 2), (4, 6, 5), 2.0, 0x7F, 0.397, (0.0, 5.0), True),        # C up to 2^31
    ((2, 2, 3), (6, 5, 6), 2.0, 0x01, 0.05, (0.0, 2.0e4), False),      # |n| up to 2^58.3
    ((2, 2, 3), (6, 5, 6), 0.01, 0x7F, 0.01, (0.0, 0.9), True),        # E below 2^-7: wide 1/E; f / E <= 0.9 / 0.001,
    # so that the masses' fixed-point sums over 180 cells stay below 2^19 (f up to 900 would exceed it)
    ((2, 3, 2), (32, 31, 2), 3.0, 0x11, 0.02, (0.0, 1.0), False),
    ((3, 2, 2), (7, 4, 11), 7.3, 0x13, 0.05, (-0.2, 0.9), True),       # central cells at 8.9e-16
    ((2, 2, 3), (6, 33, 4), 7.3, 0x01, 0.3, (0.0, 0.9), False),
    ((1, 3, 2), (35, 35, 2), 0.7, 0x03, 0.1, (0.0, 2.0), True),
    ((2, 3, 8), (6, 5, 4), 2.0, 0x12, 0.05, (-0.2, 0.9), True),        # the force by mirrored cells: z cells
    ((1, 8, 2), (26, 34, 16), 2.0, 0x7F, 0.02, (0.0, 0.9), True),      # or segments that fill the warps
    ((3, 2, 6), (6, 5, 4), 2.0, 0x12, 0.05, (-0.2, 0.9), True),        # and by rows
    ((2, 1, 1), (40, 64, 50), 2.0, 0x01, 0.02, (0.0, 0.9), False),     # several blocks for a row's 1/E
]


@pytest.mark.parametrize("nx,np_,L,mask,dt,rng,force", CASES)
def test_bits(nx, np_, L, mask, dt, rng, force):
    import torch
    from paper_1912_04457_gb300 import bz
    nxc, ns = int(np.prod(nx)), bin(mask).count("1")
    h = bz.Handle(nx=nx, dx=0.2, np_=np_, L=L, seed=3, species_mask=mask)
    h.set_force_term(force)
    cfg = O.make_config(nx=nx, dx=0.2, np_=np_, L=L, seed=3, species_mask=mask, force=force)
    st = I.encode(I.random_f(np_, ns, nxc, 33, *rng), mask)
    dev = torch.from_numpy(st.reshape(-1)).cuda()
    mom = torch.empty(nxc * ns * 5, dtype=torch.float64, device="cuda")
    out = torch.empty_like(dev)
    m2 = O.masses(cfg, st)
    h.moments(dev, mom)
    assert np.array_equal(h.get_masses(), m2)
    assert np.array_equal(mom.cpu().numpy().reshape(nxc, ns, 5), O.moments(cfg, st, m2)[0])
    h.drift(dev, out, dt)
    assert np.array_equal(out.cpu().numpy().reshape(st.shape), O.drift(cfg, st, m2, dt).reshape(st.shape))
    src = h.energy_source(dev, dt, 0.9 * m2).cpu().numpy().reshape(nxc, ns, 3)
    assert np.array_equal(src, O.energy_source(cfg, st, m2, 0.9 * m2, dt).reshape(nxc, ns, 3))


WIDE = [
    # nx, np, mask, dt (dx = 0.2), m^2 / (smallest p^2 of the grid), force: Courant numbers beyond dt/dx
    ((3, 2, 5), (6, 4, 7), 0x03, 0.19, (-0.9, -0.9), True),         # |p| / E up to 3: C above 2^30
    ((2, 3, 2), (4, 6, 8), 0x01, 0.19, (-0.9999, 0.5), False),      # and above 2^31, next to cells of m^2 > 0
    ((4, 1, 3), (4, 5, 6), 0x12, 0.3, (-0.9, 0.0), True),           # dt/dx = 1.5
    ((2, 3, 8), (6, 4, 8), 0x03, 0.19, (-0.9, -0.9), True),
    ((2, 2, 4), (4, 5, 6), 0x12, 0.3, (-0.9, 0.0), True),
    ((5, 2, 1), (4, 5, 6), 0x01, 0.3, (-0.9999, 0.0), False),
    ((2, 1, 1), (256, 256, 130), 0x01, 0.19, (-0.9999, 0.0), False),  # too many tiles: rows of p cells
]


@pytest.mark.parametrize("nx,np_,mask,dt,m2_rng,force", WIDE)
def test_negative_mass_squared(nx, np_, mask, dt, m2_rng, force):
    """A state with negative cells can have m^2 < 0, where |p| / E exceeds 1 and Courant
    numbers leave the range that dt/dx gives: the fluxes stay the exact products."""
    import torch
    from paper_1912_04457_gb300 import bz
    nxc, ns, L = int(np.prod(nx)), bin(mask).count("1"), 2.0
    pp = sum(min(abs(-L + (j + 0.5) * 2 * L / n) for j in range(n)) ** 2 for n in np_)
    kw = dict(nx=nx, dx=0.2, np_=np_, L=L, seed=3, species_mask=mask)
    cfg = O.make_config(force=force, **kw)
    # the masses are linear in f (E = |p| at the first evaluation): each x cell's largest |m^2| to a share of pp
    f = I.random_f(np_, ns, nxc, 21, 0.005, 0.01)
    share = np.linspace(m2_rng[0], m2_rng[1], nxc)
    f *= (share * pp / O.masses(cfg, I.encode(f, mask)).max(axis=1))[None, :, None]
    st = I.encode(f, mask)
    m2 = O.masses(cfg, st)
    assert m2.min() < -0.89 * pp and m2.min() > -pp
    h = bz.Handle(**kw)
    h.set_force_term(force)
    dev = torch.from_numpy(st.reshape(-1)).cuda()
    out = torch.empty_like(dev)
    h.drift(dev, out, dt)
    assert np.array_equal(h.get_masses(), m2)
    assert np.array_equal(out.cpu().numpy().reshape(st.shape), O.drift(cfg, st, m2, dt).reshape(st.shape))
