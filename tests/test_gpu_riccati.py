"""The staged Riccati kernels (csrc/riccati_seq.cu, csrc/fxp.cuh) through
prox_{alpha f} on the sizes where they change shape: sums that end at, before
and after a warp, widths that need two to five warps, more than 128 products in
a sum, one and two row groups, chains of one and of several nodes, and stages
with fewer and with more nodes than blocks.  FP64 against the oracle's KKT
projection at the tolerance of the operator tests; FP32 through one CP step
at the FP32 tolerance of tests/test_gpu_fp32.py.  Vectors far from 1, of a
wide range, zero and not finite exercise the fixed-point products."""
import numpy as np
import pytest

from tests.gpu_common import RTOL, Pair, rel_err

pytestmark = pytest.mark.gpu
TOL_FP32_T = 2e-6

SIZES = [(1, 1), (11, 5), (12, 20), (31, 1), (30, 2), (32, 1), (33, 31), (20, 44), (64, 64), (65, 63), (127, 1),
         (1, 127), (50, 20)]


def _problem(nx, nu, shape):
    from paper_2212_01110_gb300 import workloads as W
    branching = {"star_chain": [3, 1, 1], "binary": [2, 2, 1, 1, 1], "leaves": [2, 3], "wide": [400, 1]}[shape]
    anc, _ = W.tree_from_branching(branching)
    d = W.with_tree(anc, seed=nx + 7 * nu, nx=nx, nu=nu)
    rng = np.random.default_rng(nx * 131 + nu)
    n = len(anc)
    d["A"][1:] = 0.9 * W._haar_orthogonal(rng, n - 1, nx)
    d["B"][1:] = rng.standard_normal((n - 1, nx, nu)) / np.sqrt(nx)
    return Pair(d)


def _prox(p, z):
    from paper_2212_01110_gb300 import spock
    zd = p.t(z)
    out = zd.new_empty(p.gp.n_z)
    spock.spock_prox_f_dev(p.gp.handle, p.x0, p.alpha, zd, out)
    return out.cpu().numpy()


@pytest.mark.parametrize("nx,nu", SIZES)
@pytest.mark.parametrize("shape", ["star_chain", "binary", "leaves"])
def test_prox_f_sizes(nx, nu, shape):
    import torch
    from paper_2212_01110_gb300 import spock
    p = _problem(nx, nu, shape)
    rng = np.random.default_rng(1)
    z, e = rng.standard_normal(p.gp.n_z), rng.standard_normal(p.gp.n_eta)
    assert rel_err(_prox(p, z), p.cp.prox_f(z, p.d["x0"])) < RTOL
    zd, ed = p.t(z), p.t(e)
    spock.spock_cp_step_dev(p.gp.handle, p.x0, 1, p.alpha, spock.SPOCK_FP32, zd, ed)
    ref = p.cp.T(np.concatenate([z, e]), p.d["x0"])
    assert rel_err(torch.cat([zd, ed]).cpu().numpy(), ref) < TOL_FP32_T


def test_prox_f_more_nodes_than_blocks():
    p = _problem(12, 5, "wide")
    z = np.random.default_rng(2).standard_normal(p.gp.n_z)
    assert rel_err(_prox(p, z), p.cp.prox_f(z, p.d["x0"])) < RTOL


@pytest.mark.parametrize("scale", [0.0, 1e-300, 1e-30, 1e30, 1e150])
def test_prox_f_scales(scale):
    """prox_f is affine: with x0 = 0 (and s^0 left out) it scales with z."""
    p = _problem(20, 7, "star_chain")
    p.x0.zero_()
    z = np.random.default_rng(3).standard_normal(p.gp.n_z)
    one, got = _prox(p, z)[1:], _prox(p, scale * z)[1:]
    if scale == 0.0:
        assert np.all(got == 0.0)
    else:   # 1e-300: the smallest entries are not far above the denormal range
        assert np.max(np.abs(got / scale - one)) < (1e-6 if scale < 1e-200 else RTOL) * np.max(np.abs(one))


def test_prox_f_wide_range():
    """Entries over 24 orders of magnitude in one vector."""
    p = _problem(33, 31, "binary")
    rng = np.random.default_rng(4)
    z = rng.standard_normal(p.gp.n_z) * 10.0 ** rng.uniform(-18, 6, p.gp.n_z)
    assert rel_err(_prox(p, z), p.cp.prox_f(z, p.d["x0"])) < RTOL


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_prox_f_not_finite(bad):
    """A value that is not finite in the root's part reaches the states and
    inputs it is multiplied into as one that is not finite."""
    p = _problem(12, 5, "star_chain")
    z = np.random.default_rng(5).standard_normal(p.gp.n_z)
    z[1 + p.gp.n_nodes * p.gp.nx] = bad   # u^0
    out = _prox(p, z)
    x1 = out[1 + p.gp.nx:1 + 2 * p.gp.nx]
    assert not np.isfinite(x1).any()
