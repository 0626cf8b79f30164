"""Sweeps by groups of gates stop where a fixed-point state would be further from the true one
than an FP64 state: above, the default equals VQE_FLAG_FP64_SWEEPS bit for bit."""
import numpy as np
import pytest
import torch

import paper_2311_01242_gb300 as vq
import synth

pytestmark = pytest.mark.gpu


def test_number_sector_above_the_bound():
    n, k = 25, 12  # 5,200,300 states
    rng = np.random.default_rng(17)
    H = vq.Hamiltonian.from_problem_hcb(synth.random_problem(rng, n, 2 * k, 2))
    A = vq.Ansatz(n, (1 << k) - 1, [(0, 12), (3, 20), (11, 24), (0, 20), (5, 12)], hcb=True)
    assert A.info()["sector_dim"] == 5200300
    th = torch.as_tensor(rng.normal(0.0, 0.4, size=5)).cuda()
    out = []
    for flags in (0, vq.VQE_FLAG_FP64_SWEEPS):
        old = vq.set_flags(flags)
        try:
            e, g = vq.energy_grad(H, A, th)
            out.append((vq.state(A, H, th), e.clone(), g.clone()))
        finally:
            vq.set_flags(old)
    assert all(torch.equal(a, b) for a, b in zip(*out))
