"""Contexts of different size on host threads of their own: a kernel's shared-memory limit
is one value for the process, so no launch may lower it to its own need."""
import threading

import numpy as np
import pytest

import vesselmesh as vm

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("CUDA device required", allow_module_level=True)

from paper_1810_04289_gb300 import fsi  # noqa: E402

MAT = dict(rho_f=1.05, mu_f=0.035, rho_s=1.2, E_s=3.0e6, nu_s=0.45, eta_s=0.0)


@pytest.mark.parametrize("factor_mode,ordering", [(0, 1), (3, 1)])
def test_threads_factor_with_different_shared_memory(factor_mode, ordering):
    m = vm.tube_mesh(4, 6, 2, 1, seed=3)
    y = vm.poiseuille_state(m)
    jobs, errors = [], []
    for k in range(8):
        st = torch.cuda.Stream()
        with torch.cuda.stream(st):
            S = fsi.Solver(m, MAT, fsi.fsi_default_options(n_subdomains=32, ilu_level=3 * (k % 2), overlap=1 + k % 2,
                                                           factor_mode=factor_mode, ordering=ordering))
            S.set_state(y, t=0.0)
            jobs.append((S, S.vec(y), S.vec(np.ones_like(y)), S.vec(), st))
    torch.cuda.synchronize()

    def work(job):
        S, yv, r, z, st = job
        try:
            torch.cuda.set_device(0)
            for _ in range(400):
                fsi.fsi_jacobian(S.ctx, yv)
                fsi.fsi_pc_apply(S.ctx, r, z)
        except Exception as e:  # noqa: BLE001
            errors.append(e)

    ts = [threading.Thread(target=work, args=(j,)) for j in jobs]
    [t.start() for t in ts]
    [t.join() for t in ts]
    for job in jobs:
        job[0].close()
    assert not errors, errors
