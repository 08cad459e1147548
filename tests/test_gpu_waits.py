"""Bounded waits of the pipelined factorisation and of the streamed apply that run out
(a test switch of the options: copies are never issued, or a wait gives up at once): the
call ends and reports FSI_ERR_TIMEOUT, and the device and the library stay usable.
"""
import numpy as np
import pytest

import vesselmesh as vm

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("CUDA device required", allow_module_level=True)

from paper_1810_04289_gb300 import fsi  # noqa: E402

MAT = dict(rho_f=1.05, mu_f=0.035, rho_s=1.2, E_s=3.0e6, nu_s=0.45, eta_s=0.0)
TIMEOUT = 9


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("fault_test,nsub", [(3, 2), (3, 400), (4, 2), (4, 400)])
def test_factorisation_waits_that_run_out_are_reported(precision, fault_test, nsub):
    m = vm.tube_mesh(24, 16, 5, 2, seed=3)
    y = vm.poiseuille_state(m)
    r = np.random.default_rng(8).normal(size=(m.n_nodes, 7))
    out = []
    for ft, mode in ((fault_test, 0), (0, 0), (0, 3)):
        S = fsi.Solver(m, MAT, fsi.fsi_default_options(precision=precision, n_subdomains=nsub, fault_test=ft,
                                                       factor_mode=mode))
        S.set_state(y, t=0.25)
        S.jacobian(y)
        z = S.vec()
        if ft:
            with pytest.raises(fsi.FsiError) as e:
                fsi.fsi_pc_apply(S.ctx, S.vec(r), z)
            assert e.value.status == TIMEOUT
        else:
            fsi.fsi_pc_apply(S.ctx, S.vec(r), z)
            out.append(z.cpu().numpy())
        S.close()
    assert np.array_equal(out[0], out[1])      # the next context's factors: the row kernel's bits


@pytest.mark.parametrize("precision", [0, 1])
def test_a_wait_that_gave_up_is_reported_before_a_singular_pivot(precision):
    """Two problems, one subdomain each: a tube, the waits of which run out soon, and
    20,000 nodes without a tet (empty rows, singular pivots), found singular row by row
    long after. The status is the wait's, whichever was found last."""
    m = vm.tube_config("tube-12x8x4")
    k = 20000
    m.X = np.concatenate([m.X, np.c_[np.zeros((k, 2)), 100.0 + np.arange(k)]])
    m.node_tag = np.concatenate([m.node_tag, np.full(k, vm.WALL, dtype=m.node_tag.dtype)])
    m.node_problem = np.concatenate([m.node_problem, np.ones(k, dtype=m.node_problem.dtype)])
    m.inlets = [m.inlets[0], m.inlets[0]]
    S = fsi.Solver(m, MAT, fsi.fsi_default_options(precision=precision, n_subdomains=2, fault_test=3))
    y = np.zeros((m.n_nodes, 7))
    S.set_state(y, t=0.0)
    S.jacobian(y)
    with pytest.raises(fsi.FsiError) as e:
        fsi.fsi_pc_apply(S.ctx, S.vec(np.ones((m.n_nodes, 7))), S.vec())
    assert e.value.status == TIMEOUT
    S.close()


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("nsub,ordering", [(8, 1), (900, 1), (900, 2), (8, 3)])
def test_apply_waits_that_give_up_with_copies_on_their_way(precision, nsub, ordering):
    """Team, chain and ring kernels: no barrier is armed twice, the copies land before
    the block ends, and the next context's apply is the level-scheduled kernel's."""
    m = vm.tube_mesh(24, 16, 5, 2, seed=3)
    y = vm.poiseuille_state(m)
    r = np.random.default_rng(8).normal(size=(m.n_nodes, 7))
    out = []
    for ft, mode in ((5, 1), (0, 1), (0, 2)):
        S = fsi.Solver(m, MAT, fsi.fsi_default_options(precision=precision, n_subdomains=nsub, ordering=ordering,
                                                       fault_test=ft, apply_mode=mode))
        S.set_state(y, t=0.25)
        S.jacobian(y)
        z = S.vec()
        if ft:
            with pytest.raises(fsi.FsiError) as e:
                fsi.fsi_pc_apply(S.ctx, S.vec(r), z)
            assert e.value.status == TIMEOUT
        else:
            fsi.fsi_pc_apply(S.ctx, S.vec(r), z)
            out.append(z.cpu().numpy())
        S.close()
    # FP64: the row sums' order; mixed: FP32 solves of the same factors in another order
    for c in ([0, 1, 2], [3], [4, 5, 6]):
        far = np.abs(out[0][:, c] - out[1][:, c]).max() / np.abs(out[1][:, c]).max()
        assert far <= (1e-2 if precision else 1e-10), far


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("ordering", [1, 3])
def test_a_wait_that_gives_up_on_one_lane_is_reported(precision, ordering):
    m = vm.tube_mesh(24, 16, 5, 2, seed=3)
    S = fsi.Solver(m, MAT, fsi.fsi_default_options(precision=precision, n_subdomains=8, ordering=ordering,
                                                   fault_test=6))
    y = vm.poiseuille_state(m)
    S.set_state(y, t=0.25)
    S.jacobian(y)
    with pytest.raises(fsi.FsiError) as e:
        fsi.fsi_pc_apply(S.ctx, S.vec(np.ones((m.n_nodes, 7))), S.vec())
    assert e.value.status == TIMEOUT
    S.close()
