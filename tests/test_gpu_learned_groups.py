"""Learned sampler: terms of a kinematic group that share a leg (their deposits to its
cell are added before the atomic): thermal masses (groups of one and two terms), the
massless dispersion (one group of every term) and subsets of the species, against the
oracle, with the number conserved exactly."""
import numpy as np
import pytest

import oracle as O
from paper_1912_04457_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mask", [0x7F, 0x13, 0x05, 0x12])
@pytest.mark.parametrize("mass_mode", [0, 1])
def test_shared_legs(mask, mass_mode):
    import torch
    from paper_1912_04457_gb300 import bz
    np_, N, ns = (6, 4, 5), 33, bin(mask).count("1")
    h = bz.Handle(np_=np_, L=2.0, seed=9, species_mask=mask, mass_mode=mass_mode)
    cfg = O.make_config(np_=np_, L=2.0, seed=9, species_mask=mask, mass_mode=mass_mode)
    st = I.encode(I.random_f(np_, ns, 1, 5, 0.05, 0.5), mask)
    rng = np.random.default_rng(6)
    prm = np.zeros((st.size, 8), dtype=np.float32)
    prm[:, 0:3] = rng.uniform(-0.4, 0.4, (st.size, 3))
    prm[:, 3:6] = rng.uniform(0.1, 0.5, (st.size, 3))
    h.set_anchor_params(prm)
    A = torch.empty(st.size, dtype=torch.int64, device="cuda")
    h.collision_term(torch.from_numpy(st.reshape(-1)).cuda(), A, N, 2, 0.01, bz.PREC_F32, bz.SAMPLER_LEARNED)
    got = A.cpu().numpy().reshape(ns, 1, -1)
    assert int(got.sum()) == 0
    ref = O.collision(cfg, st, O.masses(cfg, st), N, step=2, dt=0.01, ubits=23, sampler=O.LEARNED,
                      prop=prm.astype(np.float64))["A"]
    # the bar of the other learned comparisons; fewer roots average a root's FP32 error (2^-20
    # of a deposit when its H is just above the re-evaluation bound) less
    assert np.linalg.norm(got - ref) <= 5e-5 * np.linalg.norm(ref.astype(np.float64))
