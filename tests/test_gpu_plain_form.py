"""FP32 collision: the form without user rows, analytic f and one-leg deposits against the
general one, which a user-defined row that no term of the species set uses selects, and
the batch's: the same deposits."""
import numpy as np
import pytest

from paper_1912_04457_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mask", [0x01, 0x02, 0x03, 0x13])
@pytest.mark.parametrize("sampler", ["symmetric", "learned"])
@pytest.mark.parametrize("N", [1, 33, 300])
def test_plain_equals_general(mask, sampler, N):
    import torch
    from paper_1912_04457_gb300 import bz
    np_, ns = (6, 5, 7) if mask != 0x01 else (8, 9, 10), bin(mask).count("1")
    st = I.encode(I.random_f(np_, ns, 2, 5, 0.05, 0.5), mask)
    rng = np.random.default_rng(6)
    prm = np.zeros((st.size, 8), dtype=np.float32)
    prm[:, 0:3] = rng.uniform(-0.4, 0.4, (st.size, 3))
    prm[:, 3:6] = rng.uniform(0.1, 0.5, (st.size, 3))
    out = []
    for user in (False, True):
        h = bz.Handle(nx=(2, 1, 1), dx=0.2, np_=np_, L=2.0, seed=9, species_mask=mask)
        if user:
            h.set_matrix_element(0, [(1.0, (0, 0, 0, 0, 0, 0))])  # q q' -> q q': needs two flavours
        if sampler == "learned":
            h.set_anchor_params(prm)
        A = torch.empty(st.size, dtype=torch.int64, device="cuda")
        h.collision_term(torch.from_numpy(st.reshape(-1)).cuda(), A, N, 2, 0.01, bz.PREC_F32,
                         bz.SAMPLER_LEARNED if sampler == "learned" else bz.SAMPLER_SYMMETRIC)
        out.append((A.cpu().numpy(), h.flags()))
    assert np.array_equal(out[0][1], out[1][1])
    assert np.array_equal(out[0][0], out[1][0])
