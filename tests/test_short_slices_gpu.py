"""Forwards of one slice of a few rows, and of short slices, on the fp32-compute path: what
a chain gets does not depend on how many chains run with it.  With few of them a frame's
features go to several CTAs, a slice of 17 to 32 rows fills half of its frame, and the
last carry leaves the running state to the caller alone."""
import pytest
import torch

import oracle
from paper_2012_11346_gb300 import slim
from paper_2012_11346_gb300 import workloads as W

from gpu_common import TOL, compare, cpu_inputs, oracle_run

pytestmark = pytest.mark.gpu

CASES = [
    # (L, C, d, M, dtype, feature)
    (17, 17, 128, 256, "f32", "relu"),   # one tile of a 32-row frame half
    (32, 64, 128, 240, "bf16", "exp"),
    (20, 64, 64, 144, "f32", "exp"),
    (25, 25, 16, 32, "f32", "relu"),
    (50, 20, 128, 256, "bf16", "relu"),  # two tiles, then one
    (33, 33, 64, 256, "f32", "exp"),     # a 48-row tile
    (130, 64, 32, 208, "f32", "exp"),
    (40, 12, 64, 192, "bf16", "exp"),    # four tiles of 16
]


@pytest.mark.parametrize("L,C,d,M,dtype,feature", CASES)
def test_a_chain_does_not_see_the_batch(cuda_device, L, C, d, M, dtype, feature):
    w = W.Workload("batch", 400, 1, L, d, M, C, dtype, feature,
                   "uniform" if feature == "relu" else "normal", "iid", seed=47)
    x = W.make_inputs(w, device=cuda_device)

    def run(n):
        return slim.forward(*(x[t][:n].contiguous() for t in "qkv"), x["omega"], C, feature, residuals=True)

    ref = run(1)
    xc = cpu_inputs({t: v[:1] if t != "omega" else v for t, v in x.items()})
    compare(dict(zip(("out", "S_state", "z_state"), ref)), oracle_run(xc, C, feature), TOL[dtype],
            names=("out", "S_state", "z_state"), where=f"{L} {C} {d} {M}", C=C)
    for n in (60, 100, 400):
        for a, b in zip(run(n), ref):
            assert torch.equal(a[:1], b), n


BIDIR = [
    # (L, C, d, M, dtype, feature): tiles of 16 and 32 rows, frames that are not full
    (6, 9, 128, 256, "bf16", "exp"),
    (14, 16, 128, 240, "f32", "relu"),
    (40, 16, 64, 144, "bf16", "exp"),
    (100, 12, 32, 64, "f32", "exp"),
    (20, 32, 64, 256, "f32", "exp"),
    (75, 30, 128, 128, "bf16", "relu"),
    (50, 20, 16, 16, "bf16", "square"),
]


@pytest.mark.parametrize("L,C,d,M,dtype,feature", BIDIR)
def test_non_causal_readout_of_short_slices(cuda_device, L, C, d, M, dtype, feature):
    w = W.Workload("batch", 400, 1, L, d, M, C, dtype, feature,
                   "uniform" if feature == "relu" else "normal", "iid", seed=53)
    x = W.make_inputs(w, device=cuda_device)
    om = None if feature == "square" else x["omega"]

    def run(n):
        return slim.forward_bidir(*(x[t][:n].contiguous() for t in "qkv"), om, C, feature)

    ref = run(1)
    xc = cpu_inputs({t: v[:1] if t != "omega" else v for t, v in x.items()})
    want = oracle.oracle_bidir_fwd(xc["q"], xc["k"], xc["v"], xc["omega"], C, feature)
    names = ("out", "S_state", "z_state")
    compare(dict(zip(names, ref)), dict(zip(names, want)), TOL[dtype], names=names,
            where=f"{L} {C} {d} {M}", C=C)
    for n in (160, 400):
        for a, b in zip(run(n), ref):
            assert torch.equal(a[:1], b), n
