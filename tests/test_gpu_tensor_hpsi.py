"""The tensor-core H psi (csrc/vqe_tc.cu) against the connectivity-row kernels
(VQE_FLAG_NO_STRINGS, FP64 multiply-adds) on the same vector: sectors whose string
counts leave ragged tiles, odd qubit and electron counts, more sources and rows
than one pass takes, one spin without electrons to move, and Hamiltonians whose
values are not symmetric under a hop's reversal, hold groups outside the
tensor-core form, or are not of the Jordan-Wigner form at all.

Tolerance: both sum the same products of a unit vector with at most a few
thousand coefficients of magnitude below 8; in FP64 that leaves an error below
1e-12 of the largest row, so 1e-11 of it separates rounding from a wrong term."""
import numpy as np
import pytest
import torch

import paper_2311_01242_gb300 as vq
import synth

pytestmark = pytest.mark.gpu


def _hf(na, nb):
    return sum(1 << (2 * i) for i in range(na)) | sum(1 << (2 * i + 1) for i in range(nb))


def _check(xs, zs, cs, n, na, nb, seed, peaked=False):
    H = vq.Hamiltonian(n, xs, zs, cs)
    A = vq.Ansatz(n, _hf(na, nb), [[0, 2 * na, -1, -1]])
    D = A.info()["sector_dim"]
    rng = np.random.default_rng(seed)
    v = rng.normal(size=D)
    if peaked:
        v *= np.exp(-rng.uniform(0.0, 30.0, size=D))  # amplitudes over thirteen decades
    v = torch.as_tensor(v / np.linalg.norm(v)).cuda()
    lam, e = vq.apply_hamiltonian_sector(H, A, v)
    old = vq.set_flags(vq.VQE_FLAG_NO_STRINGS)
    try:
        ref, e_ref = vq.apply_hamiltonian_sector(H, A, v)
    finally:
        vq.set_flags(old)
    scale = float(ref.abs().max())
    assert scale > 0.0
    assert float((lam - ref).abs().max()) <= 1e-11 * scale
    assert abs(float(e) - float(e_ref)) <= 1e-11 * max(1.0, abs(float(e_ref)))
    again, _ = vq.apply_hamiltonian_sector(H, A, v)
    assert torch.equal(lam, again)


def _molecule(n_s, seed):
    p = synth.random_problem(np.random.default_rng(seed), n_s, 2, 4)
    return vq.jordan_wigner(n_s, p.h, p.eri)


@pytest.mark.parametrize("n_s,na,nb", [(11, 5, 6), (12, 7, 4), (13, 3, 6), (14, 9, 2), (12, 6, 5)])
def test_sectors(n_s, na, nb):
    _check(*_molecule(n_s, n_s + na), 2 * n_s, na, nb, seed=nb, peaked=n_s == 12)


def test_two_passes_of_sources_and_rows():
    """16 orbitals, 6 alpha and 2 beta electrons: 66 sources (passes of 64), 136 rows (tiles of 128)."""
    _check(*_molecule(16, 4), 32, 6, 2, seed=5)


def test_odd_qubit_count():
    """23 qubits: the last alpha qubit has no beta partner."""
    xs, zs, cs = _molecule(12, 6)
    top = np.uint64(1 << 23)
    keep = ((xs & top) == 0) & ((zs & top) == 0)
    _check(xs[keep], zs[keep], cs[keep], 23, 6, 5, seed=7)


@pytest.mark.parametrize("what", ["odd", "rest", "both"])
def test_general_values_and_groups(what):
    xs, zs, cs = _molecule(12, 8)
    rng = np.random.default_rng(9)
    if what != "rest":
        cs = cs * (1.0 + 0.3 * rng.normal(size=len(cs)))  # no symmetry left between a hop's strings
    if what != "odd":
        # strings without the sign of a hop, longer than four flips, and two-spin triples
        ex = [0b101, 0b1010, 0b110011, 0b11, 0b111100001111]
        xs = np.concatenate([xs, np.array(ex * 3, dtype=np.uint64)])
        zs = np.concatenate([zs, rng.integers(0, 1 << 24, size=len(ex) * 3).astype(np.uint64)])
        cs = np.concatenate([cs, rng.normal(0.0, 0.2, size=len(ex) * 3)])
    _check(xs, zs, cs, 24, 5, 6, seed=10)


def test_non_finite_input_reaches_the_output():
    xs, zs, cs = _molecule(12, 11)
    H = vq.Hamiltonian(24, xs, zs, cs)
    A = vq.Ansatz(24, _hf(5, 6), [[0, 10, -1, -1]])
    v = torch.zeros(A.info()["sector_dim"], dtype=torch.float64, device="cuda")
    v[17] = float("inf")
    lam, e = vq.apply_hamiltonian_sector(H, A, v)
    assert not torch.isfinite(lam[17]) and not torch.isfinite(e)
