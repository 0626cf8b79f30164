"""The gate sweeps in cluster shared memory (csrc/vqe_sweep.cu) against the launches
per gate (VQE_FLAG_FP64_SWEEPS): sectors that need one to sixteen CTAs, odd electron
counts, ansatze of one gate and none, gates with more pairs than a CTA has threads,
angles 0, +-pi/2 and pi; and batches of every cluster size against single calls.

Tolerance: fixed point keeps 2^-62 of the norm per rotation and 2^-59 ||lambda|| per
gradient product, FP64 2^-53 per operation; over a few hundred gates and ||H psi|| <
100 both stay below 1e-12, so 1e-11 separates rounding from a wrong pair or sign."""
import numpy as np
import pytest
import torch

import paper_2311_01242_gb300 as vq
import synth

pytestmark = pytest.mark.gpu


def _instance(n_s, ne, m, seed, pool="uccsd"):
    rng = np.random.default_rng(seed)
    p = synth.random_problem(rng, n_s, ne, 4)
    exc = synth.uccsd_pool(2 * n_s, ne) if pool == "uccsd" else synth.upccgsd_pool(2 * n_s)
    exc = exc[rng.permutation(len(exc))[:m]]
    th = rng.normal(0.0, 0.4, size=len(exc))
    th[:4] = np.array([0.0, np.pi / 2, -np.pi / 2, np.pi])[:min(4, len(th))]
    return vq.Hamiltonian.from_problem(p), vq.Ansatz(2 * n_s, synth.hf_bitstring(ne), exc), torch.as_tensor(th).cuda()


def _per_gate(H, A, th):
    old = vq.set_flags(vq.VQE_FLAG_FP64_SWEEPS | vq.VQE_FLAG_FORCE_STREAMING)
    try:
        e, g = vq.energy_grad(H, A, th)
        return e.clone(), g.clone()
    finally:
        vq.set_flags(old)


@pytest.mark.parametrize("n_s,ne,m,pool", [(6, 5, 40, "uccsd"), (7, 7, 90, "uccsd"), (8, 9, 1, "uccsd"),
                                           (8, 8, 200, "upccgsd"), (9, 9, 120, "uccsd"), (10, 7, 100, "uccsd"),
                                           (10, 10, 60, "uccsd"), (10, 11, 30, "upccgsd"), (11, 10, 24, "uccsd")])
def test_single_instances(n_s, ne, m, pool):
    H, A, th = _instance(n_s, ne, m, seed=10 * n_s + ne, pool=pool)
    old = vq.set_flags(vq.VQE_FLAG_FORCE_STREAMING)  # the small ones would run resident
    try:
        e, g = vq.energy_grad(H, A, th)
        e, g = e.clone(), g.clone()
        only = vq.energy(H, A, th)
    finally:
        vq.set_flags(old)
    e_ref, g_ref = _per_gate(H, A, th)
    assert abs(float(e) - float(e_ref)) <= 1e-11
    assert float((g - g_ref).abs().max()) <= 1e-11
    assert float(only) == float(e)


def test_no_gates():
    H, A, th = _instance(8, 8, 0, seed=3)
    e, g = vq.energy_grad(H, A, torch.zeros(1, dtype=torch.float64, device="cuda"))
    assert g.numel() == 0
    assert abs(float(e) - float(_per_gate(H, A, torch.zeros(1, dtype=torch.float64, device="cuda"))[0])) <= 1e-11


@pytest.mark.parametrize("copies", [1, 5])
def test_batch_equals_single_calls(copies):
    """Every cluster size in one batch, few enough instances to widen the clusters and too many to."""
    insts = [_instance(n_s, ne, m, seed=100 * c + n_s) for c in range(copies)
             for n_s, ne, m in [(7, 7, 60), (8, 7, 90), (9, 9, 50), (10, 10, 40), (10, 9, 70), (11, 10, 8)]]
    hams, ans = [i[0] for i in insts], [i[1] for i in insts]
    B = vq.Batch(hams, ans)
    theta = torch.zeros(len(insts), B.max_params, dtype=torch.float64, device="cuda")
    for i, (_, _, th) in enumerate(insts):
        theta[i, :th.numel()] = th
    e, g = B.energy_grad(theta)
    only, _ = B.energy_grad(theta, with_grad=False)
    assert torch.equal(only, e)
    for i, (H, A, th) in enumerate(insts):
        e1, g1 = vq.energy_grad(H, A, th)
        assert float(e1) == float(e[i]), i
        assert torch.equal(g1, g[i, :A.n_params]), i
    old = vq.set_flags(vq.VQE_FLAG_FP64_SWEEPS)  # the same batch by launches per gate
    try:
        e2, g2 = B.energy_grad(theta)
    finally:
        vq.set_flags(old)
    assert float((e2 - e).abs().max()) <= 1e-11
    for i, (_, A, _) in enumerate(insts):
        assert float((g2[i, :A.n_params] - g[i, :A.n_params]).abs().max()) <= 1e-11
