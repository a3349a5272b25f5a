"""FP32 collision: work units that run over several anchors and rows, parts of
one anchor, anchor subsets, and momentum axes on both sides of 128 cells (the
32-bit position of k2), against the oracle on the same 23-bit uniforms (the
FP32 bar, 2e-5 relative L2; 1e-4 where a few thousand samples leave a single root
to dominate: the roots that stay in FP32 have |H| >= tau kappa^2, so 1/sqrt(H)
with some 6 roundings of kappa^2's size is off by up to 6 2^-24 / (2 tau) = 9e-5),
sum A = 0, the same bits from both schedules."""
import os

import numpy as np
import pytest

import oracle as O
from paper_1912_04457_gb300 import inputs as I

pytestmark = pytest.mark.gpu

CASES = [
    # nx, np, mask, N, stride, offset
    ((1, 1, 1), (256, 2, 4), 0x01, 64, 1, 0),      # the longest axis
    ((1, 1, 1), (130, 129, 2), 0x03, 8, 1, 0),     # just above 128
    ((1, 1, 1), (128, 127, 2), 0x01, 8, 1, 0),     # and at it
    ((3, 2, 4), (4, 3, 2), 0x01, 33, 1, 0),        # rows shorter than a unit's anchors
    ((2, 1, 2), (6, 5, 4), 0x13, 1, 1, 0),         # one sample per anchor
    ((2, 2, 1), (6, 4, 8), 0x17, 100, 7, 3),       # a subset that skips over row ends
    ((1, 1, 1), (4, 4, 4), 0x02, 1100, 1, 0),      # an anchor in several units (N > 1024)
    ((1, 1, 1), (4, 4, 4), 0x01, 64, 1 << 33, 5),  # one anchor of a stride beyond 32 bits
]


@pytest.mark.parametrize("nx,np_,mask,N,stride,offset", CASES)
def test_units(nx, np_, mask, N, stride, offset):
    import torch
    from paper_1912_04457_gb300 import bz
    nxc = int(np.prod(nx))
    h = bz.Handle(nx=nx, dx=0.2, np_=np_, L=2.0, seed=6, species_mask=mask)
    cfg = O.make_config(nx=nx, dx=0.2, np_=np_, L=2.0, seed=6, species_mask=mask)
    h.set_anchor_subset(stride, offset)
    st = I.encode(I.random_f(np_, bin(mask).count("1"), nxc, 14, 0.05, 0.5), mask)
    dev = torch.from_numpy(st.reshape(-1)).cuda()
    A, B = torch.empty_like(dev), torch.empty_like(dev)
    h.collision_term(dev, A, N, 2, 0.01, bz.PREC_F32)
    ref = O.collision(cfg, st, O.masses(cfg, st), N, step=2, dt=0.01, ubits=23, anchor_stride=stride,
                      anchor_offset=offset)["A"].reshape(-1).astype(float)
    got = A.cpu().numpy()
    assert int(got.sum()) == 0 and np.count_nonzero(got) > 0
    tol = 2e-5 if -(-dev.numel() // stride) * N > 10000 else 1e-4
    assert np.linalg.norm(got - ref) <= tol * np.linalg.norm(ref)
    try:
        for sched in ("counter", "static"):
            os.environ["BZ_F32_SCHEDULE"] = sched
            h.reset_masses()
            h.collision_term(dev, B, N, 2, 0.01, bz.PREC_F32)
            assert torch.equal(A, B), sched
    finally:
        del os.environ["BZ_F32_SCHEDULE"]


@pytest.mark.parametrize("mask,alpha,lo,hi", [(0x01, 0.3, -0.6, 0.1), (0x13, 0.3, -0.6, 0.1), (0x7F, 1.0, -0.6, 0.1),
                                              (0x7F, 5.0, -0.2, 0.15)])
@pytest.mark.parametrize("sampler", [0, 2])
def test_negative_mass_squared(mask, alpha, lo, hi, sampler):
    """A state with negative cells can have m^2 < 0, where kappa alone no longer tells which roots
    are valid.  Most valid roots then have t or u above the regulator, and flag 0 counts
    those: the oracle's number but for roots within FP32 rounding (some 1e-6 of t's terms) of
    it, fewer than 1e-4 of them."""
    import torch
    from paper_1912_04457_gb300 import bz
    np_, N, seed = (6, 5, 4), 400, 8
    h = bz.Handle(np_=np_, L=2.0, seed=seed, species_mask=mask, alpha_s=alpha)
    cfg = O.make_config(np_=np_, L=2.0, seed=seed, species_mask=mask, alpha_s=alpha)
    st = I.encode(I.random_f(np_, bin(mask).count("1"), 1, 15, lo, hi), mask)
    m2 = O.masses(cfg, st)
    assert m2[0, 0] < 0
    prop = None
    if sampler == 2:
        h.proposal_init(3)
        h.proposal_infer()
        prop = h.anchor_params().astype(np.float64)
    A = torch.empty(st.size, dtype=torch.int64, device="cuda")
    h.collision_term(torch.from_numpy(st.reshape(-1)).cuda(), A, N, 2, 0.01, bz.PREC_F32, sampler)
    want = int(O.collision(cfg, st, m2, N, step=2, dt=0.01, ubits=23, sampler=sampler, prop=prop)["flags"][0])
    assert want > 1000 and abs(int(h.flags()[0]) - want) <= 1e-4 * want
    assert int(A.sum().item()) == 0
