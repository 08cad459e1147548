"""The chain and team kernels of the preconditioner apply against the level-scheduled
kernel on the same factors, on both sides of the subdomain counts where the choice
between them changes and down to subdomains of a few nodes (Sec. 3, Eq. 16).

FP64: the kernels differ by the order of each row's sum only; 1e-10 per field group
is the bound of the oracle comparison. Mixed: both are FP32 solves with the same
factors, so each is off the FP64 apply by the error of FP32 arithmetic and of the
FP32 Jacobian on that case; the level-scheduled kernel measures it, and the chain's
may be at most twice that (plus 1e-6, for groups the error of which happens to be
small).
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
GROUPS = {"u": [0, 1, 2], "p": [3], "d": [4, 5, 6]}


@pytest.fixture(scope="module")
def case():
    m = vm.tube_mesh(24, 16, 5, 2, seed=3)
    y = vm.poiseuille_state(m)
    r = np.random.default_rng(8).normal(size=(m.n_nodes, 7))
    return m, y, r


def apply(case, precision, mode, **opt):
    m, y, r = case
    S = fsi.Solver(m, MAT, fsi.fsi_default_options(precision=precision, apply_mode=mode, **opt))
    S.set_state(y, t=0.25)
    S.jacobian(y)
    z = S.vec()
    fsi.fsi_pc_apply(S.ctx, S.vec(r), z)
    out, kind = z.cpu().numpy(), S.info().apply_kernel
    S.close()
    assert mode == 0 or kind == mode
    return out


def far(a, b):
    return {g: np.abs(a[:, c] - b[:, c]).max() / np.abs(b[:, c]).max() for g, c in GROUPS.items()}


@pytest.mark.parametrize("ilu,ordering", [(1, 1), (2, 2), (3, 0), (0, 1)])
@pytest.mark.parametrize("nsub", [2, 256, 257, 608, 609, 900])
def test_chain_and_team_match_the_level_scheduled_kernel(case, nsub, ilu, ordering):
    opt = dict(n_subdomains=nsub, ilu_level=ilu, ordering=ordering)
    ref = apply(case, 0, 2, **opt)
    d64 = far(apply(case, 0, 1, **opt), ref)
    assert all(v <= 1e-10 for v in d64.values()), d64
    level, chain = far(apply(case, 1, 2, **opt), ref), far(apply(case, 1, 1, **opt), ref)
    assert all(chain[g] <= 2 * level[g] + 1e-6 for g in GROUPS), (chain, level)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("nsub,ilu,ordering", [(1, 0, 0), (1, 3, 1), (4, 1, 2), (64, 2, 1), (305, 1, 1), (900, 2, 0)])
def test_pipelined_factors_are_the_row_kernels_bits(case, precision, nsub, ilu, ordering):
    """factor_mode 0 (pipelined) does factor_mode 3's arithmetic in its order."""
    opt = dict(n_subdomains=nsub, ilu_level=ilu, ordering=ordering)
    a, b = (apply(case, precision, 0, factor_mode=k, **opt) for k in (0, 3))
    assert np.array_equal(a, b)


@pytest.mark.parametrize("precision,nsub", [(0, 700), (0, 8), (1, 500), (1, 8)])
def test_waits_that_run_out_are_reported(case, precision, nsub):
    m, y, r = case
    S = fsi.Solver(m, MAT, fsi.fsi_default_options(precision=precision, n_subdomains=nsub, fault_test=1))
    S.set_state(y, t=0.25)
    S.jacobian(y)
    with pytest.raises(fsi.FsiError) as e:
        fsi.fsi_pc_apply(S.ctx, S.vec(r), S.vec())
    assert e.value.status == 9
    S.close()
