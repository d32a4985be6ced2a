"""The FP64 form's evaluate beside another stream's kernel of seconds that holds the SMs: same bits, whatever the wait."""
import numpy as np
import pytest

from paper_2005_12351_gb300 import synth
from test_gpu_graph_calls import host, same

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("graph", [False, True])
def test_evaluate_beside_a_long_kernel(graph):
    import torch
    from gpu_util import to_dev
    from paper_2005_12351_gb300 import fmm
    pos, S = synth.make_system(120_000, 1, "uniform", 720)
    st, other = torch.cuda.Stream(), torch.cuda.Stream()
    X, S = to_dev(pos), to_dev(S)
    big = torch.rand((1_500_000, 3), dtype=torch.float64, device="cuda")
    q = torch.rand((1_500_000, 1), dtype=torch.float64, device="cuda")
    to = torch.arange(40_000, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    t = fmm.create_tree(max_leaf=32, stream=st)
    t.set_sources(X, S, 1)
    run = t.evaluate_graph if graph else t.evaluate
    ref = host(run(6, 0.5))
    assert t.info()["tc_rows"] > 0
    for wait in (0, 3):
        held = fmm.direct_sum(big, q, 0, targets=to, stream=other)         # some two seconds on every SM
        for _ in range(wait):
            t.update_moments(S)
        assert same(host(run(6, 0.5)), ref)
        del held
    t.destroy()
