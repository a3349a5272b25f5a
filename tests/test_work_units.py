"""The collision kernels' work units: every (anchor, chunk of samples) in exactly one,
on the host (compiled as plain C++, no GPU), and calls that select no anchor on the GPU."""
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_split_covers_every_chunk_once(tmp_path):
    exe = tmp_path / "split_check"
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    r = subprocess.run(["g++", "-O2", "-std=c++17", "-I", os.path.join(cuda, "include"),
                        "-I", os.path.join(ROOT, "paper_1912_04457_gb300", "csrc"),
                        os.path.join(ROOT, "tests", "split_check.cpp"), "-o", str(exe)],
                       capture_output=True, text=True)
    if r.returncode != 0:
        pytest.fail(r.stderr)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, "exit status %d: %s" % (r.returncode, r.stdout)


@pytest.mark.gpu
@pytest.mark.parametrize("prec", [0, 1])
def test_no_anchor_selected(prec):
    """An offset beyond the last cell selects no anchor: A is zeroed, nothing else happens."""
    import torch
    from paper_1912_04457_gb300 import bz
    from paper_1912_04457_gb300 import inputs as I
    np_, mask = (6, 5, 4), 0x13
    h = bz.Handle(np_=np_, L=2.0, seed=3, species_mask=mask)
    st = torch.from_numpy(I.encode(I.random_f(np_, 3, 1, 7, 0.0, 0.6), mask).reshape(-1)).cuda()
    h.set_anchor_subset(65537, 5000)
    A = torch.full_like(st, 123)
    h.collision_term(st, A, 64, 0, 0.01, prec)
    assert int(A.abs().sum().item()) == 0
    if prec == 0:
        assert np.all(h.collision_audit(st, A, 64)[4:] == 0.0)
    assert np.all(h.flags() == 0)


@pytest.mark.gpu
@pytest.mark.parametrize("batch", [False, True])
def test_few_samples_leave_room_in_the_re_evaluation_queue(batch):
    """Heavy species (thermal masses of a large coupling, some 10 GeV in a box of 2) make every
    tenth term ill-conditioned.  The queue has room for 256 samples of every unit of an anchor, so that
    at 32 samples none of them is left to FP32."""
    import torch
    from paper_1912_04457_gb300 import bz
    from paper_1912_04457_gb300 import inputs as I
    np_, mask, alpha, N = (16, 16, 16), 0x7F, 60.0, 32
    n = I.encode(I.random_f(np_, 7, 1, 7, 0.0, 0.5), mask).reshape(-1)
    if batch:
        b = bz.Batch([dict(np_=np_, L=2.0, species_mask=mask, nsamples=N, alpha_s=alpha)] * 4)
        st = torch.from_numpy(np.tile(n, 4)).cuda()
        b.step(st, 1e-9, 1)
        assert b.flags()[3] == 0
    else:
        h = bz.Handle(np_=np_, L=2.0, seed=3, species_mask=mask, alpha_s=alpha)
        A = torch.empty(n.size, dtype=torch.int64, device="cuda")
        h.collision_term(torch.from_numpy(n).cuda(), A, N, 0, 1e-9, bz.PREC_F32)
        assert h.flags()[3] == 0 and int(A.sum().item()) == 0
