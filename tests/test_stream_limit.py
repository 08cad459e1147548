"""A stage's block count is kept in a byte: a longer stage asked for is cut, not wrapped."""
import numpy as np
import pytest

import vesselmesh as vm
from test_stream_plan import lib, plan  # noqa: F401


@pytest.mark.parametrize("most", [16, 0])       # the chain's stream; the step-ahead stream
@pytest.mark.parametrize("stage", [255, 256, 400])
def test_a_stage_holds_at_most_255_blocks(lib, most, stage):  # noqa: F811
    S = plan(lib, vm.tube_config("tube-12x8x4"), 2, 2, 1, 1 << 40, most, stage)
    for s in range(2):
        sizes = S["stage"][S["stage_off"][s]:S["stage_off"][s + 1]].astype(int)
        assert sizes.sum() == S["L_off"][s + 1] - S["L_off"][s] and sizes.max() <= 255
        ends = np.array([(int(x) >> (8 * i)) & 255 for x in S["code"][S["code_off"][s]:S["code_off"][s + 1]]
                         for i in range(4)])
        # every stage but the last is ended by an entry
        assert np.count_nonzero((ends < 128) & (ends & 64 != 0)) == len(sizes) - 1
