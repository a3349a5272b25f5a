"""FP64 collision: the warp-cooperative kernel (FP32 classification of the k1z
roots, integer bins) against the oracle, bit for bit: axes at and around 128 and 256
cells, rows shorter than a unit's anchors, subsets, one sample per anchor, an
anchor in several units, both uniform resolutions, scales of L far from 1."""
import numpy as np
import pytest

import oracle as O
from paper_1912_04457_gb300 import inputs as I

pytestmark = pytest.mark.gpu

CASES = [
    # nx, np, L, mask, mass mode, N, sampler, uniform bits, stride, offset
    ((1, 1, 1), (256, 2, 4), 2.0, 0x01, 0, 64, 0, 32, 1, 0),
    ((1, 1, 1), (130, 129, 2), 2.0, 0x03, 0, 8, 0, 23, 1, 0),
    ((3, 2, 4), (4, 3, 2), 2.0, 0x01, 0, 33, 0, 32, 1, 0),
    ((2, 1, 2), (6, 5, 4), 2.0, 0x13, 0, 1, 0, 32, 1, 0),
    ((2, 2, 1), (6, 4, 8), 2.0, 0x17, 0, 100, 1, 32, 7, 3),
    ((1, 1, 1), (4, 4, 4), 2.0, 0x02, 0, 1100, 0, 23, 1, 0),
    ((1, 1, 1), (6, 6, 6), 1e-3, 0x7F, 1, 48, 0, 32, 1, 0),
    ((1, 1, 1), (6, 6, 6), 5e3, 0x7F, 0, 48, 0, 32, 1, 0),
    ((1, 1, 1), (4, 4, 4), 2.0, 0x01, 0, 64, 0, 32, 1 << 33, 5),
]


@pytest.mark.parametrize("nx,np_,L,mask,mode,N,sampler,bits,stride,offset", CASES)
def test_bits(nx, np_, L, mask, mode, N, sampler, bits, stride, offset):
    import torch
    from paper_1912_04457_gb300 import bz
    h = bz.Handle(nx=nx, dx=0.2, np_=np_, L=L, seed=8, species_mask=mask, mass_mode=mode)
    cfg = O.make_config(nx=nx, dx=0.2, np_=np_, L=L, seed=8, species_mask=mask, mass_mode=mode)
    h.set_uniform_bits(bits)
    h.set_anchor_subset(stride, offset)
    st = I.encode(I.random_f(np_, bin(mask).count("1"), int(np.prod(nx)), 15, 0.0, 0.6), mask)
    A = torch.empty(st.size, dtype=torch.int64, device="cuda")
    h.collision_term(torch.from_numpy(st.reshape(-1)).cuda(), A, N, 2, 0.01, bz.PREC_F64, sampler)
    ref = O.collision(cfg, st, O.masses(cfg, st), N, step=2, dt=0.01, sampler=sampler, ubits=bits, anchor_stride=stride,
                      anchor_offset=offset)
    got = A.cpu().numpy()
    assert np.array_equal(got, ref["A"].reshape(-1)) and np.count_nonzero(got) > 0
    assert np.array_equal(h.flags()[:2], ref["flags"])


SCALES = [
    # L, m^2 / L^2 of (g, u, d, s), mask
    (1e-12, (0.3, 0.1, 0.1, 0.2), 0x13),
    (1e-18, (0.0, 0.0, 0.0, 0.0), 0x13),
    (1e-19, (0.3, 0.1, 0.1, 0.2), 0x13),    # p^2 leaves FP32's range
    (1e-25, (0.3, 0.1, 0.1, 0.2), 0x01),
    (4e9, (0.3, 0.1, 0.1, 0.2), 0x13),      # the square of p^2 does
    (1e20, (1e-3, 1e-6, 0.0, 1e-2), 0x13),  # p^2 itself
    (2.0, (1e3, 1e-30, 1e12, 1e20), 0x0F),  # masses far from L
]


@pytest.mark.parametrize("L,m2,mask", SCALES)
def test_bits_at_any_scale(L, m2, mask):
    """Momenta and masses far from 1 (other units than GeV): the FP32 classification
    works in units of L and keeps what leaves FP32's range."""
    import torch
    from paper_1912_04457_gb300 import bz
    np_, N, dt = (6, 5, 4), 2000, 0.05 / L
    m2 = np.array([m2]) * L * L
    h = bz.Handle(np_=np_, L=L, seed=8, species_mask=mask, mass_mode=bz.MASS_FIXED)
    h.set_masses(m2)
    cfg = O.make_config(np_=np_, L=L, seed=8, species_mask=mask, mass_mode=2)
    st = I.encode(I.random_f(np_, bin(mask).count("1"), 1, 15, 0.0, 0.6), mask)
    A = torch.empty(st.size, dtype=torch.int64, device="cuda")
    h.collision_term(torch.from_numpy(st.reshape(-1)).cuda(), A, N, 2, dt, bz.PREC_F64)
    ref = O.collision(cfg, st, m2, N, step=2, dt=dt)
    got = A.cpu().numpy()
    assert np.array_equal(got, ref["A"].reshape(-1)) and np.count_nonzero(got) > 0
    assert np.array_equal(h.flags()[:2], ref["flags"])


@pytest.mark.parametrize("mask,alpha,lo,hi", [(0x01, 0.3, -0.6, 0.1), (0x13, 0.3, -0.6, 0.1), (0x7F, 1.0, -0.6, 0.1),
                                              (0x7F, 5.0, -0.2, 0.15)])
def test_negative_mass_squared(mask, alpha, lo, hi):
    """A state with negative cells can have m^2 < 0: E^2 and a^2 may be negative, energies NaN, and
    kappa no longer tells which roots are valid.  Bit for bit the formula, its flags included."""
    import torch
    from paper_1912_04457_gb300 import bz
    np_, N = (6, 5, 4), 400
    h = bz.Handle(np_=np_, L=2.0, seed=8, species_mask=mask, alpha_s=alpha)
    cfg = O.make_config(np_=np_, L=2.0, seed=8, species_mask=mask, alpha_s=alpha)
    st = I.encode(I.random_f(np_, bin(mask).count("1"), 1, 15, lo, hi), mask)
    m2 = O.masses(cfg, st)
    assert m2[0, 0] < 0
    dev = torch.from_numpy(st.reshape(-1)).cuda()
    A = torch.empty(st.size, dtype=torch.int64, device="cuda")
    h.collision_term(dev, A, N, 2, 0.01, bz.PREC_F64)
    assert np.array_equal(h.get_masses(), m2)
    ref = O.collision(cfg, st, m2, N, step=2, dt=0.01)
    got = A.cpu().numpy()
    assert np.array_equal(got, ref["A"].reshape(-1)) and np.count_nonzero(got) > 0
    assert np.array_equal(h.flags()[:2], ref["flags"])
