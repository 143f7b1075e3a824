"""Device memory of a problem: its factors are held once per precision, in the
one layout that the staged, the direct and the single-block kernels read, so
the largest problem that fits the device is bounded by them alone."""
import pytest

pytestmark = pytest.mark.gpu


def test_factors_are_held_once():
    import torch
    from paper_2212_01110_gb300 import spock
    from paper_2212_01110_gb300 import workloads as W
    nx, nu = 50, 20
    d = W.large_tree(3, branching_stages=5, branch=4, N=8, nx=nx, nu=nu)
    n = len(d["anc"])
    nl = len(set(d["anc"][1:].tolist()))
    warm = spock.Problem(W.small_binary(0))   # module loading
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    p = spock.Problem(d)
    torch.cuda.synchronize()
    used = before - torch.cuda.mem_get_info()[0]
    # [Abar | B], its transpose; E, K, Rt^-1 and K^T: 8 + 4 bytes each
    factors = 12 * ((n - 1) * 2 * nx * (nx + nu) + nl * (3 * nu * nx + nu * nu))
    p.close()
    warm.close()
    # the rest (weights, boxes, scratch of 2 nx + 3 nu + 2 (nx + nu) numbers a
    # node, index arrays) is below a tenth of them at this size
    assert factors <= used <= 1.1 * factors + 64 * 2 ** 20, (used, factors)
