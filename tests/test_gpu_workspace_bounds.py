"""Workspace of spin sectors whose two spins have very different numbers of strings: the dense
one-spin operands of the tensor-core H psi stay in proportion, and results agree with the
kernels that do without (tolerance of test_gpu_tensor_hpsi.py: 1e-11 of the largest entry)."""
import numpy as np
import pytest
import torch

import paper_2311_01242_gb300 as vq
import synth

pytestmark = pytest.mark.gpu


def _sector(n_s, na, nb, m=6):
    p = synth.random_problem(np.random.default_rng(n_s + na), n_s, 2, 2)
    hf = sum(1 << (2 * i) for i in range(na)) | sum(1 << (2 * i + 1) for i in range(nb))
    exc = [[2 * i, 2 * a, -1, -1] for i in range(na) for a in range(na, n_s)][:m]
    th = torch.as_tensor(np.random.default_rng(3).normal(0.0, 0.4, size=len(exc))).cuda()
    return vq.Hamiltonian.from_problem(p), vq.Ansatz(2 * n_s, hf, exc), th


def test_large_square_operands():
    """12,870 x 120 strings: 2.3 GB of one-spin digits beside 50 MB of vectors."""
    H, A, th = _sector(16, 8, 2)
    D = A.info()["sector_dim"]
    assert D == 12870 * 120
    assert vq.workspace_bytes(H, A, vq.VQE_WS_ENERGY) < (2 << 30)
    v = torch.randn(D, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    lam, _ = vq.apply_hamiltonian_sector(H, A, v)
    old = vq.set_flags(vq.VQE_FLAG_NO_STRINGS)
    try:
        ref, _ = vq.apply_hamiltonian_sector(H, A, v)
    finally:
        vq.set_flags(old)
    assert float((lam - ref).abs().max()) <= 1e-11 * float(ref.abs().max())


def test_batch_of_skewed_sectors():
    """3,003 x 14 strings: in a batch each instance would hold 130 MB of digits for 42,042 states."""
    insts = [_sector(14, 6, 1, m) for m in (3, 6, 4)] + [_sector(8, 4, 4)]
    B = vq.Batch([i[0] for i in insts], [i[1] for i in insts])
    assert B.workspace_bytes(True) < 256 << 20
    theta = torch.zeros(len(insts), B.max_params, dtype=torch.float64, device="cuda")
    for i, (_, _, th) in enumerate(insts):
        theta[i, :th.numel()] = th
    e, g = B.energy_grad(theta)
    for i, (H, A, th) in enumerate(insts):
        e1, g1 = vq.energy_grad(H, A, th)
        assert float(e1) == float(e[i])
        assert torch.equal(g1, g[i, :A.n_params])


def test_energy_only_batch():
    """Without the gradient a batch holds no forward outputs (16 bytes for every amplitude pair of every
    gate), and its energies are the same, by the plan of either precision."""
    rng = np.random.default_rng(9)
    insts = []
    for n_s, ne, m in ((8, 8, 200), (9, 8, 150), (10, 10, 120)):
        exc = synth.uccsd_pool(2 * n_s, ne)
        exc = exc[rng.permutation(len(exc))[:m]]
        th = torch.as_tensor(rng.normal(0.0, 0.4, size=len(exc))).cuda()
        insts.append((vq.Hamiltonian.from_problem(synth.random_problem(rng, n_s, ne, 4)),
                      vq.Ansatz(2 * n_s, synth.hf_bitstring(ne), exc), th))
    B = vq.Batch([i[0] for i in insts], [i[1] for i in insts])
    pairs = sum(i[1].info()["n_pairs"] for i in insts)
    assert B.workspace_bytes(True) - B.workspace_bytes(False) >= 16 * pairs
    theta = torch.zeros(len(insts), B.max_params, dtype=torch.float64, device="cuda")
    for i, (_, _, th) in enumerate(insts):
        theta[i, :th.numel()] = th
    for flags in (0, vq.VQE_FLAG_FP64_SWEEPS):
        old = vq.set_flags(flags)
        try:
            e, g = [t.clone() for t in B.energy_grad(theta)]
            ws = vq.alloc_workspace(B.workspace_bytes(False))
            only = torch.zeros_like(e)
            B.energy_grad(theta, only, None, ws, with_grad=False)
            B.status(ws)
        finally:
            vq.set_flags(old)
        assert torch.equal(only, e)


def test_fp64_call_in_a_capture_before_its_plan():
    """VQE_FLAG_FP64_SWEEPS first used inside a capture: no plan can be built there, so the instances run
    one by one in the workspace sized without the flag, with the bits of single calls under it."""
    rng = np.random.default_rng(10)
    insts = []
    for n_s, ne, m in ((8, 8, 30), (9, 8, 20), (8, 7, 40)):
        exc = synth.uccsd_pool(2 * n_s, ne)
        exc = exc[rng.permutation(len(exc))[:m]]
        th = torch.as_tensor(rng.normal(0.0, 0.4, size=len(exc))).cuda()
        insts.append((vq.Hamiltonian.from_problem(synth.random_problem(rng, n_s, ne, 4)),
                      vq.Ansatz(2 * n_s, synth.hf_bitstring(ne), exc), th))
    B = vq.Batch([i[0] for i in insts], [i[1] for i in insts])
    theta = torch.zeros(len(insts), B.max_params, dtype=torch.float64, device="cuda")
    for i, (_, _, th) in enumerate(insts):
        theta[i, :th.numel()] = th
    ws = vq.alloc_workspace(B.workspace_bytes(True))
    e = torch.zeros(len(insts), dtype=torch.float64, device="cuda")
    g = torch.zeros(len(insts), B.max_params, dtype=torch.float64, device="cuda")
    old = vq.set_flags(vq.VQE_FLAG_FP64_SWEEPS)
    try:
        singles = [[t.clone() for t in vq.energy_grad(H, A, th)] for H, A, th in insts]  # loads the kernels
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            B.energy_grad(theta, e, g, ws)
        graph.replay()
        torch.cuda.synchronize()
    finally:
        vq.set_flags(old)
    for i, (e1, g1) in enumerate(singles):
        assert float(e1) == float(e[i])
        assert torch.equal(g1, g[i, :insts[i][1].n_params])
