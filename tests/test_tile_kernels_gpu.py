"""The fp32-compute path's tile kernels at the edges of their tiling: slices
that are padded to 16, 32 and 48 rows (several tiles per 64-row frame, a last
frame with fewer), feature counts that leave a part of the staged 32- and
64-feature chunks empty, the reduction groups of short tiles, one d per kernel
instantiation, and more frames than a backward launch has CTAs -- against the
fp64 oracle at the usual bounds (1e-5 fp32, 2e-2 bf16)."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2012_11346_gb300 import slim
from paper_2012_11346_gb300 import workloads as W

from gpu_common import TOL, compare, cpu_inputs, gpu_run, oracle_run

pytestmark = pytest.mark.gpu

CASES = [
    # (B, L, d, M, C, dtype, feature)
    (1, 100, 16, 80, 7, "f32", "exp"),        # 7-row slices in 16-row tiles, last frame short
    (1, 1100, 16, 16, 64, "f32", "relu"),     # two reduction groups (M = 16)
    (2, 333, 32, 32, 64, "bf16", "exp"),      # two reduction groups (M = 32)
    (1, 209, 32, 112, 33, "f32", "relu"),     # 33-row slices in 48-row tiles
    (1, 131, 64, 144, 17, "bf16", "exp"),     # 17-row slices in 32-row tiles
    (1, 203, 64, 96, 100, "f32", "exp"),      # a 36-row last tile in every slice
    (2, 321, 128, 256, 16, "bf16", "exp"),    # 8 score groups, 4 readout groups
    (1, 145, 128, 240, 48, "f32", "exp"),
    (350, 65, 16, 32, 64, "bf16", "relu"),    # frames > CTAs of the backward
]


@pytest.mark.parametrize("B,L,d,M,C,dtype,feature", CASES)
def test_tile_edges(cuda_device, B, L, d, M, C, dtype, feature):
    w = W.Workload("tiles", B, 1, L, d, M, C, dtype, feature,
                   "uniform" if feature == "relu" else "normal", "iid", seed=31)
    x = W.make_inputs(w, device=cuda_device)
    xc = cpu_inputs(x)
    compare(gpu_run(x, C, feature), oracle_run(xc, C, feature), TOL[dtype], where=w.name,
            scale=float(np.linalg.norm(xc["dout"].ravel())), C=C if B < 10 else None)


def test_noalloc_sweeps_chains_in_batches(cuda_device):
    """A forward whose full workspace exceeds slim_fwd_noalloc's scratch runs on
    fewer rows and chains at a time: the same bits as slim_fwd.  The problem size
    that it refuses does not follow the scratch's layout."""
    w = W.Workload("batches", 60, 1, 200, 64, 256, 7, "f32", "exp", "normal", "iid", seed=32)
    x = W.make_inputs(w, device=cuda_device)
    assert slim.workspace_size(60, 1, 200, 64, 256, 7, torch.float32, "exp", False) > 16 << 20
    ref = slim.forward(x["q"], x["k"], x["v"], x["omega"], w.C, w.feature, residuals=True)
    got = [torch.full_like(t, float("nan")) for t in ref]
    st = slim.library().slim_fwd_noalloc(
        x["q"].data_ptr(), x["k"].data_ptr(), x["v"].data_ptr(), x["omega"].data_ptr(), w.B, w.H,
        w.L, w.d, w.M, w.C, slim.DTYPES[torch.float32], slim.FEATURES[w.feature],
        *(t.data_ptr() for t in got), ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert st == 0
    torch.cuda.synchronize()
    for a, b in zip(got, ref):
        assert torch.equal(a, b)
    # 4 B ((1 + 2) 256 65 + 16 (4 64 + 2 256 + 2 + 16)) bytes: 16.4 MiB at B = 69
    z = [torch.zeros(69, 1, 200, 64, device=cuda_device) for _ in range(4)]
    S, zs = torch.zeros(69, 1, 256, 64, device=cuda_device), torch.zeros(69, 1, 256, device=cuda_device)
    st = slim.library().slim_fwd_noalloc(
        z[0].data_ptr(), z[1].data_ptr(), z[2].data_ptr(), x["omega"].data_ptr(), 69, 1, w.L, w.d, w.M,
        w.C, slim.DTYPES[torch.float32], slim.FEATURES[w.feature], z[3].data_ptr(), S.data_ptr(),
        zs.data_ptr(), None, None, ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert st == 3  # SLIM_ERR_WORKSPACE


SHORT = [
    # (rows per call, d, M, dtype, feature)
    (1, 64, 256, "bf16", "exp"),
    (3, 16, 48, "f32", "relu"),
    (16, 32, 112, "bf16", "relu"),
    (16, 128, 256, "f32", "exp"),
    (7, 128, 128, "bf16", "square"),
    (13, 64, 144, "f32", "exp"),
]


@pytest.mark.parametrize("r,d,M,dtype,feature", SHORT)
def test_short_calls_equal_short_slices(cuda_device, r, d, M, dtype, feature):
    """Calls of r <= 16 rows on a running state (one launch each, the state
    updated in place) against one call with slices of r rows on the general
    kernels: the same bits in out, the state and its residuals."""
    n = 5
    w = W.Workload("short", 2, 3, n * r, d, M, r, dtype, feature,
                   "uniform" if feature == "relu" else "normal", "iid", seed=33)
    x = W.make_inputs(w, device=cuda_device)
    om = None if feature == "square" else x["omega"]
    ref = slim.forward(x["q"], x["k"], x["v"], om, r, feature, residuals=True)
    S, z, S_lo, z_lo = (torch.zeros_like(t) for t in ref[1:])
    ws = torch.empty(slim.workspace_size(2, 3, r, d, M, r, x["q"].dtype, feature, False),
                     dtype=torch.uint8, device=cuda_device)
    for i in range(n):
        q, k, v = (x[t][:, :, i * r:(i + 1) * r].contiguous() for t in ("q", "k", "v"))
        out = torch.empty_like(q)
        before = slim.launch_count()
        slim.forward_into(q, k, v, om, 1000, feature, out, S, z, ws, S_lo=S_lo, z_lo=z_lo,
                          S_init=S, z_init=z, S_init_lo=S_lo, z_init_lo=z_lo)
        assert slim.launch_count() == before + 1
        assert torch.equal(out, ref[0][:, :, i * r:(i + 1) * r]), i
    for got, want in zip((S, z, S_lo, z_lo), ref[1:]):
        assert torch.equal(got, want)
