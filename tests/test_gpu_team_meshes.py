"""The team and chain applies on a tree, on a batch of uneven tubes and with two layers of
overlap, against the level-scheduled kernel on the same factors (Sec. 3, Eq. 16). The
bounds are those of tests/test_gpu_chain.py: FP64 1e-10 per field group; mixed at most
twice the level-scheduled kernel's own distance from the FP64 apply, plus 1e-6.
"""
import numpy as np
import pytest

import vesselmesh as vm

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("CUDA device required", allow_module_level=True)

from test_gpu_chain import GROUPS, apply, far  # noqa: E402


@pytest.fixture(scope="module", params=["tree", "batch", "tube"])
def case(request):
    if request.param == "tree":
        m = vm.tree_config("tree-3gen", h=0.35)
        y = np.zeros((m.n_nodes, 7))
        y[:, 2] = 10.0 * ((m.node_tag & vm.FLUID) != 0)
    elif request.param == "batch":
        parts = [vm.tube_config("tube-12x8x4"), vm.tube_mesh(24, 16, 5, 2, seed=3), vm.tube_mesh(6, 8, 2, 1, seed=9)]
        m = vm.concat_meshes(parts)
        y = np.concatenate([vm.poiseuille_state(p) for p in parts])
    else:
        m = vm.tube_mesh(24, 16, 5, 2, seed=3)
        y = vm.poiseuille_state(m)
    return m, y, np.random.default_rng(8).normal(size=(m.n_nodes, 7))


@pytest.mark.parametrize("ilu,overlap", [(1, 2), (2, 1)])
@pytest.mark.parametrize("nsub", [5, 120, 500, 700])      # both teams; FP64 team and FP32 chain; chains
def test_applies_match_the_level_scheduled_kernel(case, nsub, ilu, overlap):
    opt = dict(n_subdomains=nsub, ilu_level=ilu, overlap=overlap)
    ref = apply(case, 0, 2, **opt)
    d64 = far(apply(case, 0, 1, **opt), ref)
    assert all(v <= 1e-10 for v in d64.values()), d64
    level, chain = far(apply(case, 1, 2, **opt), ref), far(apply(case, 1, 1, **opt), ref)
    assert all(chain[g] <= 2 * level[g] + 1e-6 for g in GROUPS), (chain, level)
