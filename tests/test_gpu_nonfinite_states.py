"""H psi of vectors that hold infinities and NaN: they reach the outputs that H connects them
to and no others, in the hop kernels (csrc/vqe_hop.cu) as in the kernels that sum group by group
(VQE_FLAG_NO_STRINGS). Finite outputs: the tolerance of test_gpu_tensor_hpsi.py, 1e-11 of the
largest."""
import numpy as np
import pytest
import torch

import paper_2311_01242_gb300 as vq
import synth

pytestmark = pytest.mark.gpu


def _same(H, A, seed):
    D = A.info()["sector_dim"]
    rng = np.random.default_rng(seed)
    v = rng.normal(size=D)
    v /= np.linalg.norm(v)
    v[[0, D // 3]] = np.inf
    v[D // 2] = -np.inf
    v[D - 7] = np.nan
    v = torch.as_tensor(v).cuda()
    out = []
    for flags in (0, vq.VQE_FLAG_NO_STRINGS):
        old = vq.set_flags(flags)
        try:
            lam, e = vq.apply_hamiltonian_sector(H, A, v)
        finally:
            vq.set_flags(old)
        assert torch.isnan(e)
        out.append(lam)
    a, b = out
    fine = torch.isfinite(b)
    assert 0 < int(fine.sum()) < D
    assert torch.equal(torch.isnan(a), torch.isnan(b))
    assert torch.equal(a[~fine & ~torch.isnan(b)], b[~fine & ~torch.isnan(b)])
    assert float((a[fine] - b[fine]).abs().max()) <= 1e-11 * float(b[fine].abs().max())


@pytest.mark.parametrize("diagonal", [True, False])
@pytest.mark.parametrize("n,k", [(21, 10), (28, 6)])
def test_hops(n, k, diagonal):
    rng = np.random.default_rng(n)
    p = synth.random_problem(rng, n, 2 * k, 3)
    xs, zs, cs = vq.hcb_hamiltonian(n, p.h, p.eri, p.c0)
    if not diagonal:
        xs, zs, cs = xs[xs != 0], zs[xs != 0], cs[xs != 0]
    H = vq.Hamiltonian(n, xs, zs, cs)
    _same(H, vq.Ansatz(n, (1 << k) - 1, [(0, k)], hcb=True), n + k)


def _spin(n_s, na, nb):
    p = synth.random_problem(np.random.default_rng(100 * n_s + na), n_s, 2, 3)
    xs, zs, cs = vq.jordan_wigner(n_s, p.h, p.eri)
    hf = sum(1 << (2 * i) for i in range(na)) | sum(1 << (2 * i + 1) for i in range(nb))
    return xs, zs, cs, vq.Ansatz(2 * n_s, hf, [[0, 2 * na, -1, -1]])


@pytest.mark.parametrize("n_s,na,nb", [(12, 4, 5), (15, 1, 5), (10, 5, 5), (9, 4, 1)])
def test_tensor_core_strings(n_s, na, nb):
    """Each form of the string kernel that takes over (many, some and few beta strings)."""
    xs, zs, cs, A = _spin(n_s, na, nb)
    _same(vq.Hamiltonian(2 * n_s, xs, zs, cs), A, n_s + na)


def test_tensor_core_with_groups_outside_its_form():
    xs, zs, cs, A = _spin(12, 5, 4)
    rng = np.random.default_rng(3)
    ex = [0b101, 0b1010, 0b110011, 0b111100001111]
    xs = np.concatenate([xs, np.array(ex, dtype=np.uint64)])
    zs = np.concatenate([zs, rng.integers(0, 1 << 24, size=len(ex)).astype(np.uint64)])
    cs = np.concatenate([cs, rng.normal(0.0, 0.2, size=len(ex))])
    _same(vq.Hamiltonian(24, xs, zs, cs), A, 5)
