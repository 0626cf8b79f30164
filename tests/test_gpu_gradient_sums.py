"""Gradient sums of the fixed-point gate sweeps against long double.

Groups of gates (csrc/vqe_group.cu): the state that vqe.state returns and lambda from
apply_hamiltonian_sector are the ones that the gradient call computes, bit for bit, so the
last gate's component is known exactly: 2 sum s (lambda_k' psi_k - lambda_k psi_k'). Tolerance:
the call rounds that sum to FP64 (2^-53 of it) and lambda to 2^-62 of a bound below
2 ||lambda||; the latter errors are independent, so with ||psi|| = 1 their sum stays, at six
deviations, below 6 * 0.3 * 2^-61 * 2 ||lambda|| < 2^-58 ||lambda||. Sums of products cut off at
the fixed point's unit scatter by sqrt(pairs) units of 2^-61 ||lambda|| instead: 2^-54 and more
with 14,400 pairs.

Cluster shared memory (csrc/vqe_sweep.cu): the gradient from the state in long double, whose
distance the FP64 launches per gate must not beat."""
import numpy as np
import pytest
import torch

import paper_2311_01242_gb300 as vq
import synth
from oracle.ansatz import excitation_ops
from oracle.fermion import apply_string, popcount
from oracle.hamiltonian import sector_basis

pytestmark = pytest.mark.gpu
L = np.longdouble


def _pairs(basis, exc, hcb):
    if hcb:
        i, a = np.uint64(exc[0]), np.uint64(exc[1])
        one = np.uint64(1)
        k = basis[(((basis >> i) & one) == one) & (((basis >> a) & one) == 0)]
        kp, s = k ^ ((one << i) | (one << a)), np.ones(len(k))
    else:
        kp, s, ok = apply_string(basis, excitation_ops(exc)[0])
        k, kp, s = basis[ok], kp[ok], s[ok].astype(float)
    return np.searchsorted(basis, k), np.searchsorted(basis, kp), s


def _spin(n_s, ne, doubles, singles, seed, scale=0.4):
    rng = np.random.default_rng(seed)
    H = vq.Hamiltonian.from_problem(synth.random_problem(rng, n_s, ne, 4))
    pool = synth.uccsd_pool(2 * n_s, ne)
    sg, db = [e for e in pool if e[2] < 0], [e for e in pool if e[2] >= 0]
    exc = [db[i] for i in rng.permutation(len(db))[:doubles]] + [sg[i] for i in rng.permutation(len(sg))[:singles]]
    hf = synth.hf_bitstring(ne)
    basis = sector_basis(2 * n_s, (ne + 1) // 2, ne // 2)
    return H, vq.Ansatz(2 * n_s, hf, exc), exc, rng.normal(0.0, scale, size=len(exc)), basis, hf


def _boson(n, k, m, seed):
    rng = np.random.default_rng(seed)
    H = vq.Hamiltonian.from_problem_hcb(synth.random_problem(rng, n, 2 * k, 4))
    exc = [(i, a) for i in range(k) for a in range(k, n)]
    exc = [exc[i] for i in rng.permutation(len(exc))[:m]]
    basis = np.arange(1 << n, dtype=np.uint64)
    basis = basis[popcount(basis) == k]
    return H, vq.Ansatz(n, (1 << k) - 1, exc, hcb=True), exc, rng.normal(0.0, 0.4, size=m), basis, (1 << k) - 1


@pytest.mark.parametrize("which", ["boson 352,716", "boson 705,432", "spin 245,025", "spin 627,264"])
def test_groups_last_gate(which):
    hcb = which.startswith("boson")
    H, A, exc, th, basis, _ = {"boson 352,716": lambda: _boson(21, 10, 24, 1), "boson 705,432": lambda: _boson(22, 11, 24, 2),
                               "spin 245,025": lambda: _spin(12, 8, 24, 4, 3),
                               "spin 627,264": lambda: _spin(12, 10, 24, 4, 4)}[which]()
    assert A.info()["sector_dim"] == len(basis) == int(which.split()[1].replace(",", ""))
    t = torch.as_tensor(th).cuda()
    psi = vq.state(A, H, t)[torch.as_tensor(basis.astype(np.int64)).cuda()].real.contiguous()
    lam, e_ref = vq.apply_hamiltonian_sector(H, A, psi)
    e, g = vq.energy_grad(H, A, t)
    assert float(e) == float(e_ref)  # the same psi and lambda
    psi, lam = psi.cpu().numpy().astype(L), lam.cpu().numpy().astype(L)
    k, kp, s = _pairs(basis, exc[-1], hcb)
    ref = 2 * (s * (lam[kp] * psi[k] - lam[k] * psi[kp])).sum()
    assert abs(L(float(g[-1])) - ref) <= 2.0 ** -52 * abs(ref) + 2.0 ** -58 * np.sqrt((lam * lam).sum())


def test_cluster_sweeps_no_further_than_fp64():
    H, A, exc, th, basis, hf = _spin(10, 10, 220, 36, 1, scale=0.05)
    assert len(basis) == 63504  # cluster shared memory
    pairs = [_pairs(basis, x, False) for x in exc]
    x = np.zeros(len(basis), dtype=L)
    x[np.searchsorted(basis, np.uint64(hf))] = 1

    def turn(v, p, a):
        k, kp, s = p
        c, sn = np.cos(L(a)), np.sin(L(a)) * s
        u, w = v[k].copy(), v[kp].copy()
        v[k], v[kp] = c * u - sn * w, c * w + sn * u

    for p, a in zip(pairs, th):
        turn(x, p, a)
    lam, _ = vq.apply_hamiltonian_sector(H, A, torch.as_tensor(x.astype(np.float64)).cuda())
    y, ref = lam.cpu().numpy().astype(L), []
    for p, a in list(zip(pairs, th))[::-1]:
        k, kp, s = p
        ref.append(2 * (s * (y[kp] * x[k] - y[k] * x[kp])).sum())
        turn(x, p, -a)
        turn(y, p, -a)
    ref, t, off = np.array(ref)[::-1], torch.as_tensor(th).cuda(), []
    for flags in (0, vq.VQE_FLAG_FP64_SWEEPS):
        old = vq.set_flags(flags)
        try:
            g = vq.energy_grad(H, A, t)[1].cpu().numpy()
        finally:
            vq.set_flags(old)
        off.append(float(np.sqrt(((g - ref) ** 2).sum() / (ref ** 2).sum())))
    assert off[0] <= off[1], off
