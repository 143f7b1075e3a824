"""The staged Riccati kernels (csrc/riccati_seq.cu) where blocks take several
sequences with one or two slots of shared memory each: node blocks below and above
the size from which single nodes use two slots, sizes where two slots leave two,
one or no resident block, and numbers of sequences on both sides of the SM count
and of two per SM.  FP64 against the direct kernels, which the operator tests hold to
the oracle, at the tolerance of those tests.  FP32 sums do not depend on the
slots: bit for bit against a batch of the one problem, whose blocks take one
sequence each with one slot."""
import numpy as np
import pytest

from tests.gpu_common import RTOL, rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("branching", [[130, 1, 1], [200, 1, 1], [320, 1, 1, 1], [340, 2], [20, 20, 1]])
@pytest.mark.parametrize("nx,nu", [(12, 5), (25, 15), (33, 15), (50, 20), (64, 32), (90, 38)])
def test_sequences_per_block(nx, nu, branching, monkeypatch):
    import torch
    from paper_2212_01110_gb300 import spock
    from paper_2212_01110_gb300 import workloads as W
    anc, _ = W.tree_from_branching(branching)
    d = W.with_tree(anc, seed=nx + 7 * nu, nx=nx, nu=nu)
    rng = np.random.default_rng(nx * 131 + nu)
    n = len(anc)
    d["A"][1:] = 0.9 * W._haar_orthogonal(rng, n - 1, nx)
    d["B"][1:] = rng.standard_normal((n - 1, nx, nu)) / np.sqrt(nx)
    p = spock.Problem(d)
    alpha = 0.99 / p.norm_L
    t = lambda a: torch.tensor(np.asarray(a, float), dtype=torch.float64, device="cuda:0")
    x0, z, e = t(d["x0"]), t(rng.standard_normal(p.n_z)), t(rng.standard_normal(p.n_eta))

    def T():
        zo, eo = torch.empty_like(z), torch.empty_like(e)
        spock.spock_T_dev(p.handle, x0, alpha, z, e, zo, eo)
        return torch.cat([zo, eo]).cpu().numpy()

    monkeypatch.delenv("SPOCK_RICCATI_KERNELS", raising=False)
    got = T()
    s = spock.spock_default_settings(max_iter=0, precision=spock.SPOCK_FP32, fp64_tail=0)
    zs, es, zb, eb = z.clone(), e.clone(), z.clone(), e.clone()   # T of (z, e)
    spock.spock_solve_dev(p.handle, x0, s, zs, es, 1)
    monkeypatch.setenv("SPOCK_RICCATI_KERNELS", "staged")
    monkeypatch.setenv("SPOCK_BATCH_MODE", "list")
    batch = spock.spock_batch_create([p.handle])
    spock.spock_batch_solve_dev(batch, [x0], s, [zb], [eb], 1)
    spock.spock_free(batch)
    monkeypatch.setenv("SPOCK_RICCATI_KERNELS", "direct")
    ref = T()
    assert rel_err(got, ref) < RTOL
    assert torch.equal(zs, zb) and rel_err(zs.cpu().numpy(), ref[:p.n_z]) < 1e-4   # (a T was evaluated at all)
