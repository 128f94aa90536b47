"""slim_fwd_noalloc where the full workspace exceeds its scratch: the sweep takes the rows
that the scratch holds, not the fewest it can run in."""
import ctypes

import pytest
import torch

from paper_2012_11346_gb300 import slim
from paper_2012_11346_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,L,d,M,C,dtype", [
    (1, 5000, 128, 256, 16, "bf16"),  # short slices, four to a frame
    (1, 5000, 128, 256, 32, "bf16"),
    (4, 5000, 64, 128, 48, "f32"),    # one to a frame
    (20, 2000, 64, 128, 100, "f32"),  # long slices
    (60, 1100, 64, 256, 7, "f32"),    # in batches of chains
])
def test_sweep_fills_the_scratch(cuda_device, B, L, d, M, C, dtype):
    w = W.Workload("fill", B, 1, L, d, M, C, dtype, "exp", "normal", "iid", seed=43)
    x = W.make_inputs(w, device=cuda_device)
    assert slim.workspace_size(B, 1, L, d, M, C, x["q"].dtype, "exp", False) > 16 << 20
    ref = slim.forward(x["q"], x["k"], x["v"], x["omega"], C, "exp", residuals=True)
    got = [torch.full_like(t, float("nan")) for t in ref]
    before = slim.launch_count()
    st = slim.library().slim_fwd_noalloc(
        x["q"].data_ptr(), x["k"].data_ptr(), x["v"].data_ptr(), x["omega"].data_ptr(), B, 1, L, d, M,
        C, slim.DTYPES[x["q"].dtype], slim.FEATURES["exp"], *(t.data_ptr() for t in got),
        ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert st == 0
    launches = slim.launch_count() - before
    torch.cuda.synchronize()
    for a, b in zip(got, ref):
        assert torch.equal(a, b)
    # a 64-row frame takes its totals (a pair of them where slices share a frame), its
    # tiles' z and g(K) in pieces: the 16 MiB hold at least this many in turn, less the
    # chains' own share (a state pair and a frame each), and a last sequence of any size
    # per batch of chains
    shared = C <= 32
    frame = 4 * M * (d + 1) * (2 if shared else 1) + 4 * M * 9 * shared + 128 * M * (2 if dtype == "bf16" else 3)
    chain = 8 * M * (d + 1) + frame
    batches = -(-B * chain // (15 << 20))
    frames = B * -(-L // C) * -(-C // 64) if not shared else B * -(-L // (C * (4 if C <= 16 else 2)))
    held = ((15 << 20) - 8 * M * (d + 1) * min(B, (15 << 20) // chain)) // frame
    assert launches <= 3 * (2 * frames // held + 2 * batches) + batches, (launches, frames, held)
