"""The layer stack where slices are short, the last one above all: the segment calls on
them run in the workspace that slim_stack_workspace_size gives.  Against the oracle's
stack."""
import numpy as np
import pytest
import torch

import oracle
from paper_2012_11346_gb300 import slim
from paper_2012_11346_gb300 import workloads as W

from gpu_common import TOL, compare, oracle_run, to64

CASES = [  # d, M, dtype, feature
    (16, 32, "f32", "exp"),
    (64, 64, "bf16", "square"),
    (64, 256, "f32", "exp"),
]


def workload(d, M, dtype, feature, C, rows, B=1, H=2):
    return W.Workload("remainder", B, H, C + rows, d, M, C, dtype, feature, "normal", "iid", seed=41)


@pytest.mark.gpu
@pytest.mark.parametrize("C", [40, 64])
@pytest.mark.parametrize("rows", [1, 16, 17, 32, 33])
@pytest.mark.parametrize("d,M,dtype,feature", CASES)
def test_stack_with_a_short_last_slice(cuda_device, d, M, dtype, feature, rows, C):
    w = workload(d, M, dtype, feature, C, rows)
    layers = 2
    x = W.make_stack_inputs(w, layers, device=cuda_device)
    oms = None if feature == "square" else x["omegas"]
    y, S, z, Sl, zl = slim.stack_forward(x["x"], oms, C, feature, layers=layers)
    dx, dom = slim.stack_backward(x["x"], oms, x["dy"], S, z, C, feature, S_lo=Sl, z_lo=zl)
    xc, omc = to64(x["x"]), list(to64(x["omegas"]))
    ry, rS, rz = oracle.oracle_stack_fwd(xc, omc, C, feature)
    rdx, rdom = oracle.oracle_stack_bwd(xc, omc, to64(x["dy"]), rS, rz, C, feature)
    got = {"out": y, "S_state": S, "z_state": z, "dq": dx}
    ref = {"out": ry, "S_state": rS, "z_state": rz, "dq": rdx}
    if dom is not None:
        got["domega"], ref["domega"] = dom, rdom
    compare(got, ref, TOL[dtype], names=tuple(got), where=f"{w} {C} {rows}")


@pytest.mark.gpu
@pytest.mark.parametrize("rows,C", [(1, 64), (32, 40)])
def test_relu_stack_with_a_short_last_slice(cuda_device, rows, C):
    """One layer, whose oracle gets the library's own inputs u, rounded as the library
    rounds them: a ReLU decision can follow that rounding.  dy is zero outside the last slice."""
    w = workload(32, 64, "f32", "relu", C, rows)
    x = W.make_stack_inputs(w, 1, device=cuda_device)
    x["dy"][:, :, :C] = 0
    y, S, z, Sl, zl = slim.stack_forward(x["x"], x["omegas"], C, "relu", layers=1)
    _, dom = slim.stack_backward(x["x"], x["omegas"], x["dy"], S, z, C, "relu", S_lo=Sl, z_lo=zl)
    xf = x["x"].double()
    u = to64((xf * w.d ** -0.25 / torch.sqrt((xf * xf).mean(-1, keepdim=True) + 1e-6)).float())
    ref = oracle_run({"q": u, "k": u, "v": u, "omega": to64(x["omegas"][0]), "dout": to64(x["dy"])},
                     C, "relu")
    got = {"S_state": S[0], "z_state": z[0], "domega": dom[0]}
    compare(got, ref, TOL["f32"], names=tuple(got), where=f"relu {rows} {C}")


@pytest.mark.gpu
@pytest.mark.parametrize("rows", [1, 17])
def test_short_last_slice_of_many_chains(cuda_device, rows):
    """Tensor-core slices: the last slice's backward has its own kernel, whose workspace is the
    one that counts (512 chains, where another kernel's would be larger)."""
    w = W.WORKLOADS["L4096_bf16"].with_(B=64, H=8, L=64 + rows, C=64, M=128)
    x = W.make_stack_inputs(w, 1, device=cuda_device)
    y, S, z, Sl, zl = slim.stack_forward(x["x"], x["omegas"], w.C, w.feature)
    keep = [(0, 0), (63, 7)]
    dy = torch.zeros_like(x["dy"])
    for b, h in keep:
        dy[b, h] = x["dy"][b, h]
    dx, dom = slim.stack_backward(x["x"], x["omegas"], dy, S, z, w.C, w.feature, S_lo=Sl, z_lo=zl)
    omc, ref_dom = list(to64(x["omegas"])), 0.0
    for b, h in keep:
        xc = to64(x["x"][b:b + 1, h:h + 1])
        ry, rS, rz = oracle.oracle_stack_fwd(xc, omc, w.C, w.feature)
        rdx, rdom = oracle.oracle_stack_bwd(xc, omc, to64(dy[b:b + 1, h:h + 1]), rS, rz, w.C, w.feature)
        ref_dom = ref_dom + rdom
        got = {"out": y[b:b + 1, h:h + 1], "S_state": S[:, b:b + 1, h:h + 1],
               "z_state": z[:, b:b + 1, h:h + 1], "dq": dx[b:b + 1, h:h + 1]}
        ref = {"out": ry, "S_state": rS, "z_state": rz, "dq": rdx}
        compare(got, ref, TOL["bf16"], names=tuple(got), where=f"chain ({b},{h})")
    compare({"domega": dom}, {"domega": np.asarray(ref_dom)}, TOL["bf16"], names=("domega",))


@pytest.mark.gpu
@pytest.mark.parametrize("C,L,M", [(48, 128, 256), (33, 67, 128), (16, 41, 256)])
def test_stack_of_short_slices(cuda_device, C, L, M):
    """Every slice has fewer than 64 rows (the short kernel serves them all)."""
    w = W.WORKLOADS["L4096_bf16"].with_(B=1, H=2, L=L, C=C, M=M)
    x = W.make_stack_inputs(w, 2, device=cuda_device)
    y, S, z, Sl, zl = slim.stack_forward(x["x"], x["omegas"], C, w.feature)
    dx, dom = slim.stack_backward(x["x"], x["omegas"], x["dy"], S, z, C, w.feature, S_lo=Sl, z_lo=zl)
    xc, omc = to64(x["x"]), list(to64(x["omegas"]))
    ry, rS, rz = oracle.oracle_stack_fwd(xc, omc, C, w.feature)
    rdx, rdom = oracle.oracle_stack_bwd(xc, omc, to64(x["dy"]), rS, rz, C, w.feature)
    got = {"out": y, "S_state": S, "z_state": z, "dq": dx, "domega": dom}
    ref = {"out": ry, "S_state": rS, "z_state": rz, "dq": rdx, "domega": rdom}
    compare(got, ref, TOL["bf16"], names=tuple(got), where=f"{C} {L} {M}")
