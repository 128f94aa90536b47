"""The layer stack's last slice when it has fewer than 64 rows: its backward has
its own kernel on the bf16 path, at every padded height (16, 32, 48 and 64 rows) and
both feature counts, against the oracle's stack."""
import pytest
import torch

import oracle
from paper_2012_11346_gb300 import slim
from paper_2012_11346_gb300 import workloads as W

from gpu_common import TOL, compare, to64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,M,feature", [(1, 256, "exp"), (16, 128, "exp"), (17, 256, "relu"),
                                            (33, 256, "exp"), (48, 128, "relu"), (63, 256, "exp")])
def test_short_last_slice(cuda_device, rows, M, feature):
    w = W.WORKLOADS["L4096_bf16"].with_(B=1, H=3, L=128 + rows, C=128, M=M, feature=feature)
    x = W.make_stack_inputs(w, 2, device=cuda_device)
    y, S, z, Sl, zl = slim.stack_forward(x["x"], x["omegas"], w.C, feature, layers=2)
    dx, dom = slim.stack_backward(x["x"], x["omegas"], x["dy"], S, z, w.C, feature, S_lo=Sl, z_lo=zl)
    xc, omc = to64(x["x"]), list(to64(x["omegas"]))
    ry, rS, rz = oracle.oracle_stack_fwd(xc, omc, w.C, feature)
    rdx, rdom = oracle.oracle_stack_bwd(xc, omc, to64(x["dy"]), rS, rz, w.C, feature)
    got = {"out": y, "S_state": S, "z_state": z, "dq": dx, "domega": dom}
    ref = {"out": ry, "S_state": rS, "z_state": rz, "dq": rdx, "domega": rdom}
    compare(got, ref, TOL["bf16"], names=tuple(got), where=f"tail {rows} {M} {feature}")
