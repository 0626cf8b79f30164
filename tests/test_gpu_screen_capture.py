"""ADAPT screening captured straight after vqe_pool_workspace_bytes takes the route of every
later call: the tables of the gate groups are built when the workspace is sized, not by the
first call, which cannot build them under capture."""
import numpy as np
import pytest
import torch

import paper_2311_01242_gb300 as vq
import synth

pytestmark = pytest.mark.gpu


def test_captured_first_call():
    rng = np.random.default_rng(31)
    n_s, ne = 12, 8  # 245,025 states: sweeps by groups
    H = vq.Hamiltonian.from_problem(synth.random_problem(rng, n_s, ne, 3))
    exc = synth.uccsd_pool(2 * n_s, ne)
    hf = synth.hf_bitstring(ne)
    pool = vq.Ansatz(2 * n_s, hf, exc)
    first, A = (vq.Ansatz(2 * n_s, hf, exc[rng.permutation(len(exc))[:24]]) for _ in range(2))
    th = torch.as_tensor(rng.normal(0.0, 0.4, size=24)).cuda()
    vq.pool_gradients(H, first, pool, th)  # loads the kernels
    ws = vq.alloc_workspace(vq.pool_workspace_bytes(H, A, pool))
    out = (torch.zeros(1, dtype=torch.float64, device="cuda"), torch.zeros(len(exc), dtype=torch.float64, device="cuda"))
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        vq.pool_gradients(H, A, pool, th, workspace=ws, out=out)
    graph.replay()
    torch.cuda.synchronize()
    e, g = out[0].clone(), out[1].clone()
    vq.pool_gradients(H, A, pool, th, workspace=ws, out=out)
    assert torch.equal(e, out[0]) and torch.equal(g, out[1])
