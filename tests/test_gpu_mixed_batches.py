"""Batches whose instances take different routes or launch shapes, against single calls
bit for bit (every route promises that)."""
import numpy as np
import pytest
import torch

import paper_2311_01242_gb300 as vq
import synth

pytestmark = pytest.mark.gpu


def _instance(n_s, ne, m, seed):
    rng = np.random.default_rng(seed)
    p = synth.random_problem(rng, n_s, ne, 4)
    exc = synth.uccsd_pool(2 * n_s, ne)
    exc = exc[rng.permutation(len(exc))[:m]]
    th = rng.normal(0.0, 0.4, size=len(exc))
    return vq.Hamiltonian.from_problem(p), vq.Ansatz(2 * n_s, synth.hf_bitstring(ne), exc), torch.as_tensor(th).cuda()


def _batch(insts):
    B = vq.Batch([i[0] for i in insts], [i[1] for i in insts])
    theta = torch.zeros(len(insts), B.max_params, dtype=torch.float64, device="cuda")
    for i, (_, _, th) in enumerate(insts):
        theta[i, :th.numel()] = th
    return B, theta


def _equal_single_calls(insts, e, g):
    for i, (H, A, th) in enumerate(insts):
        e1, g1 = vq.energy_grad(H, A, th)
        assert float(e1) == float(e[i]), i
        assert torch.equal(g1, g[i, :A.n_params]), i


def test_large_state_beside_many_threads():
    """Cluster sweeps on one CTA each: 11,025 states and 884 gates leave shared memory for 256
    threads' copies, the other instance's gates (493 pairs each) want 512 threads. One launch
    serves both, so its threads have to fit beside both."""
    insts = [_instance(15, 4, 884, seed=21), _instance(8, 8, 360, seed=22)]
    assert [i[1].info()["sector_dim"] for i in insts] == [11025, 4900]
    B, theta = _batch(insts)
    _equal_single_calls(insts, *B.energy_grad(theta))
