"""An angle that is not finite makes the energy and every gradient component NaN, also where
the gate sweeps run in fixed point (cluster shared memory at 16 qubits, larger at 24)."""
import numpy as np
import pytest
import torch

import paper_2311_01242_gb300 as vq
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("value", [float("nan"), float("inf")])
@pytest.mark.parametrize("n_s", [8, 12])
def test_angles_that_are_not_finite(n_s, value):
    rng = np.random.default_rng(3)
    p = synth.random_problem(rng, n_s, n_s, 3)
    exc = synth.uccsd_pool(2 * n_s, n_s)[:20]
    H, A = vq.Hamiltonian.from_problem(p), vq.Ansatz(2 * n_s, synth.hf_bitstring(n_s), exc)
    th = torch.full((20,), 0.1, dtype=torch.float64, device="cuda")
    th[7] = value
    e, g = vq.energy_grad(H, A, th)
    assert np.isnan(float(e)) and torch.isnan(g).all()
