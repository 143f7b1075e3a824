"""FP64 accuracy of the staged Riccati kernels entry by entry on data whose states
and inputs differ in scale: mixed units (x = D x', u = S u', so A = D A' D^-1,
B = D B' S^-1), and two decoupled subsystems of very different magnitude.  A
format that rounds a matrix or a vector relative to its largest entry loses the
small entries there; the other tests compare relative to the largest entry of
the whole result and cannot see it.

Dynamics: every entry of x^c = A^c x + B^c u holds to the rounding of double
arithmetic.  With Abar = A + B K (formed with nu products), u = K x + d and
x^c = Abar x + B d (nx and nx + nu products), each sum of m products off by at
most (m + 1) unit roundoffs of the sum of absolute values, the residual is below
2 (nx + nu + 2) 2^-53 (|A| |x| + |B| (|K| |x| + |d| + |u|)); twice that is
asserted, for K is formed here by a factorisation of its own.

Trajectories: against the direct kernels, relative to each state's and input's
own largest value.  On the sizes taken FP64 evaluations of the recursions differ
from extended precision by at most 4.5e-14 over 8 seeds and ratios 1e4 to 1e12
(NumPy, both forms of the backward step); 1e-11 is asserted."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
TOL_TRAJECTORY = 1e-11


def _data(nx, nu, branching, ratio, decoupled=False):
    from paper_2212_01110_gb300 import workloads as W
    anc, _ = W.tree_from_branching(branching)
    n = len(anc)
    rng = np.random.default_rng(nx * 131 + nu)
    A = 0.9 * W._haar_orthogonal(rng, n, nx)
    B = rng.standard_normal((n, nx, nu)) / np.sqrt(nx)
    scale = lambda k: ratio ** rng.permutation(np.linspace(-0.5, 0.5, k)) if k > 1 else np.ones(1)  # noqa: E731
    if decoupled:   # the magnitudes in the vectors alone
        hx, hu = (nx + 1) // 2, (nu + 1) // 2
        Dx, Du = np.where(np.arange(nx) < hx, ratio, 1.0), np.where(np.arange(nu) < hu, ratio, 1.0)
        A = A * (Dx[:, None] == Dx) / 0.9
        B = B * (Dx[:, None] == Du)
    else:
        Dx, Du = scale(nx), scale(nu)
        A, B = Dx[:, None] * A / Dx, Dx[:, None] * B / Du
    d = W.with_tree(anc, seed=nx + 7 * nu, nx=nx, nu=nu)
    d["A"][1:], d["B"][1:] = A[1:], B[1:]
    nl = n - int(np.prod(branching))
    z = rng.standard_normal((n, nx)) * Dx, rng.standard_normal((nl, nu)) * Du
    return d, A, B, rng.standard_normal(nx) * Dx, z


def _gains(anc, A, B):
    """K of every nonleaf node."""
    n, nx, nu = B.shape
    kids = [np.flatnonzero(np.asarray(anc) == i) for i in range(n)]
    P, K = [None] * n, {}
    for i in range(n - 1, -1, -1):
        if len(kids[i]) == 0:
            P[i] = np.eye(nx)
            continue
        Rt = np.eye(nu) + sum(B[c].T @ P[c] @ B[c] for c in kids[i])
        s = 1.0 / np.sqrt(np.diag(Rt))   # unit diagonal before the solve
        K[i] = -s[:, None] * np.linalg.solve(s[:, None] * Rt * s, s[:, None] * sum(B[c].T @ P[c] @ A[c] for c in kids[i]))
        P[i] = np.eye(nx) + K[i].T @ K[i]
        for c in kids[i]:
            Ab = A[c] + B[c] @ K[i]
            P[i] = P[i] + Ab.T @ P[c] @ Ab
        P[i] = 0.5 * (P[i] + P[i].T)
    return kids, K


def _trajectory(d, x0, z, nx, nu):
    import torch
    from paper_2212_01110_gb300 import spock
    p = spock.Problem(d)
    f = dict(dtype=torch.float64, device="cuda:0")
    n, nl = z[0].shape[0], z[1].shape[0]
    zd = torch.zeros(p.n_z, **f)
    zd[1:1 + n * nx] = torch.tensor(z[0].ravel(), **f)
    zd[1 + n * nx:1 + n * nx + nl * nu] = torch.tensor(z[1].ravel(), **f)
    out = torch.empty_like(zd)
    spock.spock_prox_f_dev(p.handle, torch.tensor(x0, **f), 0.1, zd, out)
    o = out.cpu().numpy()
    p.close()
    return o[1:1 + n * nx].reshape(n, nx), o[1 + n * nx:1 + n * nx + nl * nu].reshape(nl, nu)


def _worst_residual(d, A, B, x, u):
    kids, K = _gains(d["anc"], A, B)
    nx, nu = B.shape[1:]
    L = np.longdouble
    worst = 0.0
    for i in K:
        free = np.abs(u[i] - K[i] @ x[i])   # d
        for c in kids[i]:
            r = np.abs(x[c].astype(L) - A[c].astype(L) @ x[i].astype(L) - B[c].astype(L) @ u[i].astype(L))
            s = np.abs(A[c]) @ np.abs(x[i]) + np.abs(B[c]) @ (np.abs(K[i]) @ np.abs(x[i]) + free + np.abs(u[i]))
            worst = max(worst, float(np.max(r / np.maximum(s, 1e-290))))
    return worst / (2 * (nx + nu + 2) * 2.0 ** -53)


@pytest.mark.parametrize("ratio", [1e4, 1e6, 1e8, 1e12])
@pytest.mark.parametrize("nx,nu,branching", [(6, 2, [2, 1, 1, 1]), (20, 7, [3, 1, 1]), (12, 5, [2, 2, 1, 1, 1]),
                                             (33, 31, [2, 2]), (50, 20, [2, 3, 1]), (64, 64, [2, 1]), (6, 2, [400, 1])])
def test_dynamics_in_mixed_units(nx, nu, branching, ratio):
    d, A, B, x0, z = _data(nx, nu, branching, ratio)
    x, u = _trajectory(d, x0, z, nx, nu)
    assert _worst_residual(d, A, B, x, u) <= 2.0


@pytest.mark.parametrize("ratio", [1e10, 1e14, 1e20])
@pytest.mark.parametrize("nx,nu,branching", [(6, 2, [2, 1, 1, 1]), (20, 7, [3, 1, 1]), (50, 20, [2, 3, 1])])
def test_dynamics_of_decoupled_subsystems(nx, nu, branching, ratio):
    d, A, B, x0, z = _data(nx, nu, branching, ratio, decoupled=True)
    x, u = _trajectory(d, x0, z, nx, nu)
    assert _worst_residual(d, A, B, x, u) <= 2.0


@pytest.mark.parametrize("ratio", [1e4, 1e6, 1e8, 1e12])
@pytest.mark.parametrize("nx,nu,branching", [(6, 1, [2, 2, 1, 1]), (13, 1, [2, 1, 1]), (24, 1, [3, 1]),
                                             (6, 2, [2, 1, 1, 1]), (20, 2, [2, 1, 1])])
def test_trajectories_in_mixed_units(nx, nu, branching, ratio, monkeypatch):
    d, A, B, x0, z = _data(nx, nu, branching, ratio)
    x, u = _trajectory(d, x0, z, nx, nu)
    monkeypatch.setenv("SPOCK_RICCATI_KERNELS", "direct")
    xr, ur = _trajectory(d, x0, z, nx, nu)
    assert np.all(np.abs(x - xr).max(0) <= TOL_TRAJECTORY * np.abs(xr).max(0))
    assert np.all(np.abs(u - ur).max(0) <= TOL_TRAJECTORY * np.abs(ur).max(0))
