"""Row sums of the mixed-precision SpMV: FP32 values and vector, each block's product in
FP32, the block products accumulated in FP64, both row mappings.

The vectors have one power of two per node and zeros elsewhere, so that every block
product is one FP32 value times a power of two, exact in FP32, and what is left is the sum
over the row's blocks. Any order of n - 1 FP64 additions is off by at most
(n - 1) u sum |p| / (1 - (n - 1) u), u = 2^-53, below n u sum |p|; a sum in pairs of floats
exceeds that in part of the rows and overflows beyond FP32's range.
"""
import math

import numpy as np
import pytest

import vesselmesh as vm

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("CUDA device required", allow_module_level=True)

from paper_1810_04289_gb300 import fsi  # noqa: E402

MAT = dict(rho_f=1.05, mu_f=0.035, rho_s=1.2, E_s=3.0e6, nu_s=0.45, eta_s=0.0)


@pytest.fixture(scope="module", params=[16, 32])
def operator(request):
    m = vm.tube_config("tube-12x8x4")
    rng = np.random.default_rng(0)
    y = vm.poiseuille_state(m)
    y = y + rng.normal(size=y.shape) * np.array([2, 2, 2, 5, 1e-4, 1e-4, 1e-4])
    y[:, 0:4] *= ((m.node_tag & vm.FLUID) != 0)[:, None]
    S = fsi.Solver(m, MAT, fsi.fsi_default_options(precision=1, n_subdomains=4, threads_per_row=request.param))
    S.set_state(y, t=0.25)
    S.jacobian(y)
    rp, col, vals = fsi.fsi_jacobian_export(S.ctx)
    yield S, np.asarray(rp), np.asarray(col), np.asarray(vals).reshape(-1, 7, 7)
    S.close()


def product(S, x):
    z = S.vec()
    fsi.fsi_spmv(S.ctx, S.vec(x), z)
    return z.cpu().numpy()


@pytest.mark.parametrize("emax", [4, 20])
def test_block_products_are_summed_in_fp64(operator, emax):
    S, rp, col, vals = operator
    n = len(rp) - 1
    rng = np.random.default_rng(3)
    k = rng.integers(0, 7, size=n)
    v = np.ldexp(rng.choice([-1.0, 1.0], size=n), rng.integers(-emax, emax + 1, size=n))
    x = np.zeros((n, 7))
    x[np.arange(n), k] = v
    z = product(S, x)
    p = vals[np.arange(len(col)), :, k[col]] * v[col][:, None]      # [blocks][component], exact
    assert np.array_equal(p, p.astype(np.float32))
    for i in range(n):
        q = p[rp[i]:rp[i + 1]]
        for r in range(7):
            bound = len(q) * 2.0 ** -53 * math.fsum(np.abs(q[:, r]))
            assert abs(z[i, r] - math.fsum(q[:, r])) <= bound, (i, r)


def test_row_sums_beyond_the_range_of_fp32_stay_finite(operator):
    S, rp, col, vals = operator
    n, done = len(rp) - 1, 0
    for i in range(0, n, 29):
        A = vals[rp[i]:rp[i + 1]]
        r = int(np.abs(A).max(axis=2).min(axis=0).argmax())          # the component with the largest smallest block
        k = np.abs(A[:, r]).argmax(axis=1)
        a = A[np.arange(len(A)), r, k]
        if np.abs(a).min() < 1.0 or len(A) < 13:
            continue
        x = np.zeros((n, 7))
        x[col[rp[i]:rp[i + 1]], k] = np.sign(a) * np.ldexp(1.0, 127 - np.frexp(np.abs(a))[1])
        p = a * x[col[rp[i]:rp[i + 1]], k]                           # in [2^126, 2^127)
        assert p.min() >= 2.0 ** 126 and p.max() < 2.0 ** 127
        z = product(S, x)[i, r]
        assert abs(z - math.fsum(p)) <= len(p) * 2.0 ** -53 * math.fsum(p)
        done += 1
    assert done > 0
