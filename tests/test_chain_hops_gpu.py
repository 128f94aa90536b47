"""The tensor-core path passes chain prefixes warp by warp for up to 40 chains and
through one flag per tile above: the same sums, so the same bits per chain."""
import pytest
import torch

from paper_2012_11346_gb300 import slim
from paper_2012_11346_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,C,M,feature", [(300, 64, 256, "exp"), (700, 256, 128, "exp"),
                                           (129, 128, 256, "relu"), (1000, 100, 128, "relu")])
def test_hops_by_warp_equal_hops_by_group(cuda_device, L, C, M, feature):
    w = W.Workload("hops", 41, 1, L, 64, M, C, "bf16", feature,
                   "uniform" if feature == "relu" else "normal", "iid", seed=41)
    x = W.make_inputs(w, device=cuda_device)
    assert slim.path_for(41, 1, L, 64, M, C, torch.bfloat16, feature) == 1

    def run(n):
        q, k, v, do = (x[t][:n].contiguous() for t in ("q", "k", "v", "dout"))
        f = slim.forward(q, k, v, x["omega"], C, feature, residuals=True)
        b = slim.backward(q, k, v, x["omega"], f[0], do, f[1], f[2], C, feature,
                          S_lo=f[3], z_lo=f[4])
        torch.cuda.synchronize()
        return [*f[:3], *b[:3]]

    for a, b in zip(run(40), run(41)):
        assert torch.equal(a, b[:40])
