"""The Gram-Schmidt norm taken inside the dots launch (orth = 0) at cycle lengths past
the default 30: more than 32 columns (two entries per lane in the scalar kernels) and
the longest cycle, 64 columns, the dots of which fill all nine groups of vectors.

A GMRES solve on the FP64 operator reaches a relative residual of 1e-10 only if the
Arnoldi relation holds to about that accuracy; the solver's test is on the true residual.
The six-sweep form (orth = 2) is the measure of the iterations: a norm that were off
would cost at least a restart, which here is a whole cycle.
"""
import pytest

import vesselmesh as vm

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("CUDA device required", allow_module_level=True)

from test_gpu_parity import _solve_fp64_operator  # noqa: E402


@pytest.mark.parametrize("restart", [33, 64])
def test_norm_inside_the_dots_on_long_cycles(restart):
    m = vm.tube_config("tube-12x8x4")
    st2, _ = _solve_fp64_operator(m, orth=2, gmres_restart=restart)
    for fault_test in (0, 2):
        st0, _ = _solve_fp64_operator(m, orth=0, gmres_restart=restart, fault_test=fault_test)
        for st in (st2, st0):
            assert st.converged == 1 and st.rnorm <= 1e-10 * st.rnorm0 * 1.0001
        assert st0.iterations < st2.iterations + restart, (st2.iterations, st0.iterations)
