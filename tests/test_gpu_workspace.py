"""Plans in a device workspace that the caller owns (GPU): the same boxes and counters as in one
of the plan's own, run after run."""

import numpy as np
import pytest

from paper_1802_00330_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("count", [1, 3])
def test_plan_in_the_callers_tensor(count):
    torch = pytest.importorskip("torch")
    from paper_1802_00330_gb300 import _binding as B

    systems = synth.config_batched(count, seed=77, n_range=(4, 5))
    opts = {"max_results": 1 << 14}
    tensor = torch.empty(256 << 20, dtype=torch.uint8, device="cuda")
    own = B.Plan(systems, opts=opts, wave_children=1 << 17)
    theirs = B.Plan(systems, opts=opts, wave_children=1 << 17, workspace=tensor)
    try:
        own.run()
        for _ in range(2):
            theirs.run()
            for k in range(count):
                a, b = own.result(k), theirs.result(k)
                for key in ("lo", "hi", "flags", "depth"):
                    assert np.array_equal(a[key], b[key]), key
                for key in ("boxes", "hs_applied", "accepted", "split", "depth_boxes"):
                    assert np.array_equal(a["stats"][key], b["stats"][key]), key
    finally:
        own.close()
        theirs.close()


def test_too_small_a_tensor_is_refused():
    torch = pytest.importorskip("torch")
    from paper_1802_00330_gb300 import _binding as B

    tensor = torch.empty(1 << 16, dtype=torch.uint8, device="cuda")
    with pytest.raises(B.IvsError):
        B.Plan([synth.config_n2()], workspace=tensor)
