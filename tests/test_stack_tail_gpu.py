"""The layer stack's last slice when it has fewer than 64 rows: its backward has
its own kernel on the bf16 path, at every padded height (16, 32, 48 and 64 rows) and
both feature counts, against the oracle's stack."""
import pytest
import torch

import oracle
from paper_2012_11346_gb300 import slim
from paper_2012_11346_gb300 import workloads as W

from gpu_common import TOL, compare, oracle_run, to64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,M", [(1, 256), (16, 128), (33, 256), (63, 256)])
def test_short_last_slice(cuda_device, rows, M):
    feature = "exp"
    w = W.WORKLOADS["L4096_bf16"].with_(B=1, H=3, L=128 + rows, C=128, M=M, feature=feature)
    x = W.make_stack_inputs(w, 2, device=cuda_device)
    y, S, z, Sl, zl = slim.stack_forward(x["x"], x["omegas"], w.C, feature, layers=2)
    dx, dom = slim.stack_backward(x["x"], x["omegas"], x["dy"], S, z, w.C, feature, S_lo=Sl, z_lo=zl)
    xc, omc = to64(x["x"]), list(to64(x["omegas"]))
    ry, rS, rz = oracle.oracle_stack_fwd(xc, omc, w.C, feature)
    rdx, rdom = oracle.oracle_stack_bwd(xc, omc, to64(x["dy"]), rS, rz, w.C, feature)
    got = {"out": y, "S_state": S, "z_state": z, "dq": dx, "domega": dom}
    ref = {"out": ry, "S_state": rS, "z_state": rz, "dq": rdx, "domega": rdom}
    compare(got, ref, TOL["bf16"], names=tuple(got), where=f"tail {rows} {M}")


@pytest.mark.parametrize("rows,M", [(17, 256), (48, 128)])
def test_short_last_slice_relu(cuda_device, rows, M):
    """One layer, so that the oracle sees the library's own inputs: a ReLU decision
    follows the rounding of u to bf16, which the oracle's stack does not make.  dy is
    zero outside the last slice."""
    w = W.WORKLOADS["L4096_bf16"].with_(B=1, H=3, L=128 + rows, C=128, M=M, feature="relu")
    x = W.make_stack_inputs(w, 1, device=cuda_device)
    x["dy"][:, :, :128] = 0
    y, S, z, Sl, zl = slim.stack_forward(x["x"], x["omegas"], w.C, "relu", layers=1)
    _, dom = slim.stack_backward(x["x"], x["omegas"], x["dy"], S, z, w.C, "relu", S_lo=Sl, z_lo=zl)
    xf = x["x"].float()
    u = to64((xf * w.d ** -0.25 / torch.sqrt((xf * xf).mean(-1, keepdim=True) + 1e-6)).to(x["x"].dtype))
    ref = oracle_run({"q": u, "k": u, "v": u, "omega": to64(x["omegas"][0]), "dout": to64(x["dy"])},
                     w.C, "relu")
    got = {"S_state": S[0], "z_state": z[0], "domega": dom[0]}
    compare(got, ref, TOL["bf16"], names=tuple(got), where=f"tail relu {rows} {M}")
