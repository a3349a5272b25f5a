"""Homogeneous grids: the fused launches of a step (masses with the state's copy and
conversion, moments summed by the last chunk, replayed graphs) against the separate
launches that a profiled handle makes, bit for bit, and the moments against the
oracle.  Grids of one mass chunk and several, chunk edges, one moments chunk and
many, every mass mode, both precisions."""
import numpy as np
import pytest

import oracle as O
from paper_1912_04457_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("np_,mask", [((2, 1, 1), 1), ((8, 8, 4), 0x01), ((3, 86, 1), 0x13), ((16, 16, 16), 0x7F),
                                      ((17, 20, 19), 0x01), ((24, 25, 26), 0x05)])
@pytest.mark.parametrize("mass_mode", [0, 1, 2])
def test_fused_equals_separate(np_, mask, mass_mode):
    import torch
    from paper_1912_04457_gb300 import bz
    ns, npc = bin(mask).count("1"), int(np.prod(np_))
    st = I.encode(I.random_f(np_, ns, 1, 4, -0.05, 0.7), mask)
    for prec, N, nsteps in ((bz.PREC_F32, 8, 7), (bz.PREC_F64, 2, 2)):
        out = []
        for prof in (True, False):
            h = bz.Handle(np_=np_, L=2.0, seed=3, species_mask=mask, mass_mode=mass_mode)
            if mass_mode == 2:
                h.set_masses(np.full((1, 4), 0.2))
            h.profile(prof)
            dev = torch.from_numpy(st.reshape(-1).copy()).cuda()
            mom = torch.empty(nsteps * ns * 5, dtype=torch.float64, device="cuda")
            first = torch.empty(ns * 5, dtype=torch.float64, device="cuda")
            for _ in range(2):  # the second call starts where the counters of the first ended
                h.step(dev, 0.002, nsteps, N, prec, step0=5, moments_out=mom)
            h.moments(dev, first)
            out.append((dev.cpu().numpy(), mom.cpu().numpy(), first.cpu().numpy(), h.get_masses()))
        for a, b in zip(*out):
            assert np.array_equal(a, b)
        cfg = O.make_config(np_=np_, L=2.0, seed=3, species_mask=mask, mass_mode=mass_mode)
        ref = O.moments(cfg, out[1][0].reshape(ns, 1, npc), out[1][3])[0]
        assert np.array_equal(out[1][2].reshape(ref.shape), ref)
