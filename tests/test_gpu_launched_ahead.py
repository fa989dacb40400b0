"""fp32 kernels that start on the call's inputs while the kernel before them runs: steps back to back, with different inputs, give the
bits of steps that are waited for -- few items, about one an SM (148), several an SM, many rounds."""
import pytest
import torch

import paper_2608_28158_b200 as H
from parity_util import plan_of, to_physical
from workloads import make_forest, make_inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("par,off,lens,heads", [([-1], [0], [40], 1), ([-1, 0, 0], [0, 100, 33], [300, 200, 185], 1), ([-1, 0, 1, 2, 3], [0, 900, 64, 65, 7], [1100] * 5, 2),
                                               ([-1] + [0] * 30, [0] + [9 * i + 1 for i in range(30)], [2000] + [70] * 30, 8)])
def test_steps_back_to_back(par, off, lens, heads):
    fo = make_forest([(par, off, lens)])
    plan = plan_of(fo).upload()
    ws = H.Workspace(plan, heads, 64, 64, torch.float32)
    inputs = [to_physical(plan, make_inputs(fo.n_tokens, heads, 64, 64, "fp32", seed)) for seed in (51, 52)]
    step = lambda p: H.run_fwd_bwd(plan, ws, p["q"], p["k"], p["v"], p["g"], p["dO"])  # noqa: E731
    alone = []
    for p in inputs:
        alone.append(step(p))
        torch.cuda.synchronize()
    back = [step(inputs[i % 2]) for i in range(12)]
    H.harts_la_check(ws.dev_status)
    for i, out in enumerate(back):
        for n in out:
            assert torch.equal(out[n], alone[i % 2][n]), (i, n)
