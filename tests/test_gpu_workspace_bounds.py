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
