"""Sectors at the ends of the ranges of the group sweeps (csrc/vqe_group.cu), the hop kernels
(csrc/vqe_hop.cu) and the persistent launch (csrc/vqe_batch.cu): few and many particles, one
spin nearly empty, electron-number sectors with fermionic signs, Hamiltonians with groups
outside the tensor-core form. Every case states its dimension: the routes are chosen by it.

Tolerance: fixed point keeps 2^-62 of the norm per rotation, FP64 2^-53 per operation; over a
few hundred gates and ||H psi|| < 1000 both stay below 1e-11, so 1e-10 separates rounding from
a wrong pair or sign."""
import numpy as np
import pytest
import torch

import paper_2311_01242_gb300 as vq
import synth

pytestmark = pytest.mark.gpu


def _agree(H, A, th, flags):
    e, g = [t.clone() for t in vq.energy_grad(H, A, th)]
    assert float(vq.energy(H, A, th)) == float(e)
    for f in flags:
        old = vq.set_flags(f)
        try:
            e1, g1 = vq.energy_grad(H, A, th)
            assert abs(float(e1) - float(e)) <= 1e-10
            assert float((g1 - g).abs().max()) <= 1e-10
        finally:
            vq.set_flags(old)


@pytest.mark.parametrize("n,k,gates,dim", [(28, 6, 60, 376740), (32, 6, 7, 906192), (30, 24, 9, 593775)])
def test_boson_sectors(n, k, gates, dim):
    rng = np.random.default_rng(n)
    H = vq.Hamiltonian.from_problem_hcb(synth.random_problem(rng, n, 2 * k, 4))
    exc = [(i, a) for i in range(k) for a in range(k, n)]
    exc = [exc[i] for i in rng.permutation(len(exc))[:gates]]
    A = vq.Ansatz(n, (1 << k) - 1, exc, hcb=True)
    assert A.info()["sector_dim"] == dim > 262144
    th = torch.as_tensor(rng.normal(0.0, 0.4, size=gates)).cuda()
    _agree(H, A, th, [vq.VQE_FLAG_FP64_SWEEPS, vq.VQE_FLAG_NO_STRINGS])


@pytest.mark.parametrize("n_s,ne,m,dim", [(14, 6, 30, 132496), (11, 12, 20, 213444)])
def test_spin_sectors(n_s, ne, m, dim):
    rng = np.random.default_rng(n_s)
    H = vq.Hamiltonian.from_problem(synth.random_problem(rng, n_s, ne, 3))
    exc = synth.uccsd_pool(2 * n_s, ne)
    exc = exc[rng.permutation(len(exc))[:m]]
    A = vq.Ansatz(2 * n_s, synth.hf_bitstring(ne), exc)
    assert A.info()["sector_dim"] == dim > 131072
    _agree(H, A, torch.as_tensor(rng.normal(0.0, 0.4, size=m)).cuda(), [vq.VQE_FLAG_FP64_SWEEPS])


def test_electron_number_sector_with_signs():
    """Excitations that flip spins: the sector is that of the electron number, the gates carry
    fermionic signs, and H psi has groups of every form."""
    rng = np.random.default_rng(22)
    n_s, ne = 11, 8
    H = vq.Hamiltonian.from_problem(synth.random_problem(rng, n_s, ne, 3))
    exc = [[0, 9, -1, -1], [3, 8, -1, -1], [0, 2, 9, 12], [1, 6, 13, 20], [7, 21, -1, -1], [2, 5, 10, 14], [4, 7, 11, 13]]
    A = vq.Ansatz(2 * n_s, (1 << ne) - 1, exc)
    assert A.info()["sector_dim"] == 319770  # of 22 qubits, 8 electrons: no spin sector
    _agree(H, A, torch.as_tensor(rng.normal(0.0, 0.4, size=len(exc))).cuda(), [vq.VQE_FLAG_FP64_SWEEPS])


def test_batch_of_string_driven_instances():
    """Groups that the tensor cores do not take keep mid-size sectors on the real string kernels: in a
    batch persistent slots, bit for bit the single calls, for every launch shape; singles against the
    sum group by group."""
    insts = []
    for n_s, ne, m, seed in ((8, 8, 40, 1), (9, 9, 25, 2), (8, 7, 30, 3)):
        rng = np.random.default_rng(seed)
        p = synth.random_problem(rng, n_s, ne, 3)
        xs, zs, cs = vq.jordan_wigner(n_s, p.h, p.eri)
        ex = [0b101, 0b1010, 0b110011, 0b111100001111]
        xs = np.concatenate([xs, np.array(ex, dtype=np.uint64)])
        zs = np.concatenate([zs, rng.integers(0, 1 << (2 * n_s), size=len(ex)).astype(np.uint64)])
        cs = np.concatenate([cs, rng.normal(0.0, 0.2, size=len(ex))])
        exc = synth.uccsd_pool(2 * n_s, ne)
        exc = exc[rng.permutation(len(exc))[:m]]
        A = vq.Ansatz(2 * n_s, synth.hf_bitstring(ne), exc)
        insts.append((vq.Hamiltonian(2 * n_s, xs, zs, cs), A, torch.as_tensor(rng.normal(0.0, 0.4, size=m)).cuda()))
    B = vq.Batch([i[0] for i in insts], [i[1] for i in insts])
    theta = torch.zeros(len(insts), B.max_params, dtype=torch.float64, device="cuda")
    for i, (H, A, th) in enumerate(insts):
        theta[i, :th.numel()] = th
        _agree(H, A, th, [vq.VQE_FLAG_NO_STRINGS])
    gates = sum(i[1].n_params for i in insts)
    for shape in ((0, 1024, 128), (1, 256, 128), (2, 4096, 128)):
        B.set_tuning(*shape)
        assert B.tuning()["n_tasks"] > 2 * gates  # a task at least for each gate and direction
        e, g = B.energy_grad(theta)
        for i, (H, A, th) in enumerate(insts):
            e1, g1 = vq.energy_grad(H, A, th)
            assert float(e1) == float(e[i]) and torch.equal(g1, g[i, :A.n_params]), (shape, i)
