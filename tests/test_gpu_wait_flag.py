"""A kernel whose bounded wait for a bulk copy gives up sets its problem's flag
and carries on with what the buffers hold.  Every call that runs such kernels
has to report the flag as an error of its own, not as a success whose result is
wrong, and leave it cleared.  The flag is raised from the host."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def state():
    import torch
    from paper_2212_01110_gb300 import spock
    from paper_2212_01110_gb300 import workloads as W
    d = W.random_tree(4, N=6, max_branch=3, nx=5, nu=2, chain_after=2)
    p = spock.Problem(d)
    f = dict(dtype=torch.float64, device="cuda:0")
    s = {"p": p, "x0": torch.tensor(d["x0"], **f), "z": torch.zeros(p.n_z, **f), "eta": torch.zeros(p.n_eta, **f),
         "oz": torch.zeros(p.n_z, **f), "oeta": torch.zeros(p.n_eta, **f),
         "g": torch.zeros(d["nx"], **f), "batch": spock.spock_batch_create([p.handle])}
    yield s
    spock.spock_free(s["batch"])
    p.close()


def _calls(precision_bits):
    from paper_2212_01110_gb300 import spock
    prec = spock.SPOCK_FP64 if precision_bits == 64 else spock.SPOCK_FP32
    settings = spock.spock_default_settings(precision=prec, max_iter=3, fp64_tail=0)
    null = None
    return {
        "cp": lambda s: spock.spock_cp_step_dev(s["p"].handle, s["x0"], 2, 0.0, prec, s["oz"], s["oeta"]),
        "solve": lambda s: spock.spock_solve_dev(s["p"].handle, s["x0"], settings, s["oz"], s["oeta"], 0),
        "batch": lambda s: spock.spock_batch_solve_dev(s["batch"], [s["x0"]], settings, [s["oz"]], [s["oeta"]], 0),
        "prox_f": lambda s: spock.spock_prox_f_dev(s["p"].handle, s["x0"], 0.1, s["z"], s["oz"]),
        "noalloc": lambda s: spock.spock_prox_f_noalloc_dev(s["p"].handle, s["x0"], 0.1, s["z"], s["oz"]),
        "T": lambda s: spock.spock_T_dev(s["p"].handle, s["x0"], 0.1, s["z"], s["eta"], s["oz"], s["oeta"]),
        "grad": lambda s: spock.spock_grad_dev(s["p"].handle, s["z"], s["eta"], prec, s["g"], null, null, null, null,
                                               null),
        "adjoint": lambda s: spock.spock_adjoint_dev(s["p"].handle, s["z"], s["eta"], None, 2, 1e-8, s["g"], null,
                                                     null, null, null, null),
    }


@pytest.mark.parametrize("bits", [64, 32])
@pytest.mark.parametrize("name", ["cp", "solve", "batch", "prox_f", "noalloc", "T", "grad", "adjoint"])
def test_flag_is_the_calls_own_error(state, name, bits):
    from paper_2212_01110_gb300 import spock
    call = _calls(bits)[name]
    lib = C.CDLL(spock.LIB_PATH)
    lib.spock_internal_raise_wait_flag.argtypes = [C.c_void_p]
    call(state)   # plans and workspaces
    assert lib.spock_internal_raise_wait_flag(state["p"].handle) == 0
    with pytest.raises(spock.SpockError) as e:
        call(state)
    assert e.value.code == -5 and "timed out" in str(e.value)
    call(state)   # the flag is cleared
    assert np.isfinite(state["oz"].cpu().numpy()).all()
