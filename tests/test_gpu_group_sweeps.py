"""The gate sweeps by groups (csrc/vqe_group.cu) against the launches per gate
(VQE_FLAG_FP64_SWEEPS), and H psi by hops (csrc/vqe_hop.cu) against the connectivity
rows (VQE_FLAG_NO_STRINGS): spin and electron-number sectors, low and odd electron
counts, one gate, repeated gates and gates that no state allows.

Tolerance: fixed point keeps 2^-62 of the norm per rotation and 2^-61 ||lambda|| per
gradient product, FP64 2^-53 per operation; over a few hundred gates and ||H psi|| <
1000 both stay below 1e-11, so 1e-10 separates rounding from a wrong pair or sign."""
import numpy as np
import pytest
import torch

import paper_2311_01242_gb300 as vq
import synth

pytestmark = pytest.mark.gpu


def _hcb(n, pairs, exc, seed):
    rng = np.random.default_rng(seed)
    p = synth.random_problem(rng, n, 2 * pairs, 4)
    A = vq.Ansatz(n, (1 << pairs) - 1, exc, hcb=True)
    th = torch.as_tensor(rng.normal(0.0, 0.4, size=len(exc))).cuda()
    return vq.Hamiltonian.from_problem_hcb(p), A, th


def _both(H, A, th, flag):
    out = []
    for f in (0, flag):
        old = vq.set_flags(f)
        try:
            e, g = vq.energy_grad(H, A, th)
            out.append((float(e), g.clone(), float(vq.energy(H, A, th))))
        finally:
            vq.set_flags(old)
    return out


@pytest.mark.parametrize("n_s,ne,m", [(11, 10, 40), (11, 11, 1), (12, 8, 75), (12, 11, 33), (13, 6, 50)])
def test_spin_sectors(n_s, ne, m):
    rng = np.random.default_rng(n_s * 100 + ne)
    p = synth.random_problem(rng, n_s, ne, 3)
    exc = synth.uccsd_pool(2 * n_s, ne)
    exc = exc[rng.permutation(len(exc))[:m]]
    exc = np.concatenate([exc, exc[:3]])  # the same gates again
    th = rng.normal(0.0, 0.4, size=len(exc))
    th[:4] = np.array([0.0, np.pi / 2, -np.pi / 2, np.pi])[:min(4, len(th))]
    H, A = vq.Hamiltonian.from_problem(p), vq.Ansatz(2 * n_s, synth.hf_bitstring(ne), exc)
    (e, g, only), (e1, g1, _) = _both(H, A, torch.as_tensor(th).cuda(), vq.VQE_FLAG_FP64_SWEEPS)
    assert only == e
    assert abs(e - e1) <= 1e-10
    assert float((g - g1).abs().max()) <= 1e-10


@pytest.mark.parametrize("n,pairs,gates", [(21, 10, 30), (22, 11, 121), (26, 6, 60), (32, 5, 7), (30, 25, 9)])
def test_number_sectors(n, pairs, gates):
    exc = [(i, a) for i in range(pairs) for a in range(pairs, n)][:gates]
    H, A, th = _hcb(n, pairs, exc, seed=n)
    (e, g, only), (e1, g1, _) = _both(H, A, th, vq.VQE_FLAG_FP64_SWEEPS)
    assert only == e
    assert abs(e - e1) <= 1e-10 and float((g - g1).abs().max()) <= 1e-10
    (_, _, _), (e2, g2, _) = _both(H, A, th, vq.VQE_FLAG_NO_STRINGS)
    assert abs(e - e2) <= 1e-10 and float((g - g2).abs().max()) <= 1e-10
