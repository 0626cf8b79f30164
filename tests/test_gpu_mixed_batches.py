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


def _boson(n, k, m, seed):
    rng = np.random.default_rng(seed)
    p = synth.random_problem(rng, n, 2 * k, 4)
    exc = [(i, a) for i in range(k) for a in range(k, n)][:m]
    th = torch.as_tensor(rng.normal(0.0, 0.4, size=len(exc))).cuda()
    return vq.Hamiltonian.from_problem_hcb(p), vq.Ansatz(n, (1 << k) - 1, exc, hcb=True), th


@pytest.fixture(scope="module")
def routes():
    """Two persistent slots (boson sectors too large for the resident kernel), two instances swept in
    cluster shared memory, one evaluated by itself (245,025 states) and one resident."""
    insts = [_boson(18, 9, 20, 1), _instance(8, 8, 40, 2), _instance(12, 8, 6, 3), _boson(18, 8, 12, 4),
             _instance(9, 8, 30, 5), _instance(4, 4, 8, 6)]
    return insts, *_batch(insts)


def test_all_routes_in_one_batch(routes):
    insts, B, theta = routes
    e, g = [t.clone() for t in B.energy_grad(theta)]
    _equal_single_calls(insts, e, g)
    only, _ = B.energy_grad(theta, with_grad=False)
    assert torch.equal(only, e)
    for shape in ((1, 256, 128), (2, 4096, 64)):
        B.set_tuning(*shape)
        assert B.tuning()["grid"] > 0
        _equal_single_calls(insts, *B.energy_grad(theta))
    B.set_tuning(0, 1024, 128)


@pytest.mark.parametrize("which", ["slot", "forward sweep", "reverse sweep", "H psi"])
def test_any_wait_that_runs_out_is_reported(routes, which):
    """Whichever kind of wait runs out, the status reports it and every output of the persistent launch
    and of the cluster sweeps is NaN; instances evaluated otherwise keep their outputs."""
    insts, B, theta = routes
    e_ref, g_ref = [t.clone() for t in B.energy_grad(theta)]
    sweeps = 2  # instances swept in cluster shared memory: two sweeps each, then one H psi for all
    queued = B.tuning()["n_tasks"] - (2 * sweeps + 1)
    task = {"slot": queued // 2, "forward sweep": queued, "reverse sweep": queued + 2 * sweeps - 1,
            "H psi": queued + 2 * sweeps}[which]
    ws = vq.alloc_workspace(B.workspace_bytes(True))
    e, g = torch.zeros_like(e_ref), torch.zeros_like(g_ref)
    B.set_wait(budget_ns=2_000_000, probe_task=task)
    try:
        B.energy_grad(theta, e, g, ws)
        with pytest.raises(vq.VQEError) as ex:
            B.status(ws)
        assert ex.value.code == 4 and "ran out" in str(ex.value)
    finally:
        B.set_wait(2_000_000_000, -1)
    for i in (0, 1, 3, 4):
        assert torch.isnan(e[i]) and torch.isnan(g[i, :insts[i][1].n_params]).all(), i
    for i in (2, 5):
        assert torch.equal(e[i], e_ref[i]) and torch.equal(g[i, :insts[i][1].n_params], g_ref[i, :insts[i][1].n_params])
    B.energy_grad(theta, e, g, ws)
    B.status(ws)
    _equal_single_calls(insts, e, g)


def test_fp64_sweeps_run_together(routes):
    """Under VQE_FLAG_FP64_SWEEPS every streamed instance that fits a persistent slot is one (H psi
    on the tensor cores between the two halves of the queue), with the bits of single calls under
    that flag, for every launch shape, without the gradient, and with a wait that runs out."""
    insts, B, theta = routes
    plain, _ = [t.clone() for t in B.energy_grad(theta)]
    old = vq.set_flags(vq.VQE_FLAG_FP64_SWEEPS)
    try:
        gates = sum(insts[i][1].n_params for i in (0, 1, 2, 3, 4))  # all but the resident one
        assert B.tuning()["n_tasks"] > 2 * gates
        for shape in ((0, 1024, 128), (1, 256, 128)):
            B.set_tuning(*shape)
            e, g = [t.clone() for t in B.energy_grad(theta)]
            _equal_single_calls(insts, e, g)
        B.set_tuning(0, 1024, 128)
        only, _ = B.energy_grad(theta, with_grad=False)
        assert torch.equal(only, e)
        ws = vq.alloc_workspace(B.workspace_bytes(True))
        n = B.tuning()["n_tasks"]
        for task in (0, n // 3, n - 2, n - 1):  # the last is H psi
            e2, g2 = torch.zeros_like(e), torch.zeros_like(g)
            B.set_wait(budget_ns=2_000_000, probe_task=task)
            try:
                B.energy_grad(theta, e2, g2, ws)
                with pytest.raises(vq.VQEError) as ex:
                    B.status(ws)
                assert ex.value.code == 4
            finally:
                B.set_wait(2_000_000_000, -1)
            assert torch.isnan(e2[[0, 1, 2, 3, 4]]).all() and torch.equal(e2[5], e[5]), task
        B.energy_grad(theta, e2, g2, ws)
        B.status(ws)
        _equal_single_calls(insts, e2, g2)
    finally:
        vq.set_flags(old)
    again, _ = B.energy_grad(theta)
    assert torch.equal(again, plain)
    # a workspace sized without the flag serves a call under it
    small = vq.alloc_workspace(B.workspace_bytes(True))
    old = vq.set_flags(vq.VQE_FLAG_FP64_SWEEPS)
    try:
        e3, g3 = torch.zeros_like(e), torch.zeros_like(g)
        B.energy_grad(theta, e3, g3, small)
        _equal_single_calls(insts, e3, g3)
    finally:
        vq.set_flags(old)
