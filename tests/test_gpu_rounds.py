"""The device-driven rounds' Gram solve (csrc/rounds_body.cuh: L D L^T in one
warp, run by the commit kernel's last block) against the host-driven loop's
Cholesky factorisation (csrc/supermann.cu), over the Anderson memories it
takes: no column, one, odd sizes, the largest; and with more columns than the
problem has directions, where columns are left out.  Both drivers take the same
branches and return the same iterate.  Tolerance: on these instances a
perturbation of one unit roundoff per evaluation of T grows by less than 1e3 in
25 iterations (tests/test_oracle_fp32_noise.py), which is 1e-13 in FP64; four
decades are left for the larger memories."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
TOL = 1e-9


def _solve(d, driver, memory, monkeypatch, iters):
    import ctypes
    import torch
    from paper_2212_01110_gb300 import spock
    monkeypatch.setenv("SPOCK_DRIVER", driver)
    P = spock.Problem(d)
    x0 = torch.tensor(d["x0"], dtype=torch.float64, device="cuda:0")
    z = torch.zeros(P.n_z, dtype=torch.float64, device="cuda:0")
    e = torch.zeros(P.n_eta, dtype=torch.float64, device="cuda:0")
    trace = np.full(2 * iters, -1, np.int32)
    s = spock.spock_default_settings(memory=memory, max_iter=iters, eps_abs=1e-13, eps_rel=1e-13)
    s.trace = trace.ctypes.data_as(ctypes.POINTER(ctypes.c_int32))
    spock.spock_solve_dev(P.handle, x0, s, z, e, 0)
    out = torch.cat([z, e]).cpu().numpy()
    P.close()
    return out, trace


@pytest.mark.parametrize("memory", [0, 1, 2, 5, 8, 13, 16])
def test_gram_solve_against_host_driver(memory, monkeypatch):
    from paper_2212_01110_gb300 import workloads as W
    d = W.random_tree(4, N=6, max_branch=3, nx=5, nu=2, chain_after=2)
    a, ta = _solve(d, "graph", memory, monkeypatch, 25)
    b, tb = _solve(d, "host", memory, monkeypatch, 25)
    assert np.array_equal(ta, tb)
    assert np.max(np.abs(a - b)) <= TOL * max(1.0, np.max(np.abs(b)))


def test_gram_solve_singular(monkeypatch):
    """A two-node problem has fewer directions than columns."""
    from paper_2212_01110_gb300 import workloads as W
    d = W.with_tree(W.tree_from_branching([1])[0], seed=11, nx=1, nu=1)
    a, _ = _solve(d, "graph", 16, monkeypatch, 12)
    assert np.isfinite(a).all()
