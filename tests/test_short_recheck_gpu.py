"""Calls of up to 16 rows against the general kernels where ReLU's recheck bound decides:
projections that lie exactly on the bound of one order of summing |omega|^2 and above the
bound of another."""
import numpy as np
import pytest
import torch

from paper_2012_11346_gb300 import slim

D, M = 64, 256
f32 = np.float32


def fma(a, b, c):
    return f32(np.float64(a) * np.float64(b) + np.float64(c))  # the product is exact in fp64


def norm_sequential(o):
    s = f32(0)
    for x in o:
        s = fma(x, x, s)
    return np.sqrt(s)


def norm_warp(o):
    """Strided terms per lane, then a butterfly."""
    s = [f32(0)] * 32
    for j, x in enumerate(o):
        s[j % 32] = fma(x, x, s[j % 32])
    for k in (16, 8, 4, 2, 1):
        s = [f32(s[i] + s[i ^ k]) for i in range(32)]
    return np.sqrt(s[0])


def on_the_bound(rng):
    """x = (1, 1, 1, 1, 0 ...) and omegas whose rounded projection is the larger of the two
    bounds; the exact projection is another number."""
    x = np.zeros(D, f32)
    x[:4] = 1
    gamma = f32(f32(2 * (D + 2)) * f32(5.9604645e-08))
    oms, n = [], 0
    while len(oms) < M:
        o = rng.standard_normal(D).astype(f32)
        o[0], o[2], o[3] = 1, -1, 0
        o[1] = f32(gamma * norm_warp(o) * f32(2) * f32(1 + 1e-4 * rng.standard_normal()))

        def bounds(o):
            return [f32(f32(gamma * f(o)) * f32(2)) for f in (norm_sequential, norm_warp)]

        a, b = bounds(o)
        c = f32(f32(f32(1) + o[1]) - f32(1))  # what is left of o[1] after 1 + o[1] - 1
        o[3] = f32(max(a, b) - c)
        if f32(c + o[3]) == max(bounds(o)) and bounds(o) == [a, b]:
            n += a != b and c != o[1]
            oms.append(o)
    return x, np.stack(oms), n


@pytest.mark.gpu
def test_recheck_bound_as_in_the_general_kernels(cuda_device):
    x, om, n = on_the_bound(np.random.default_rng(7))
    assert n > 20
    rows = torch.zeros(1, 1, 2, D, device=cuda_device)
    rows[0, 0, 0] = torch.from_numpy(x)
    om = torch.from_numpy(om).to(cuda_device)
    one = rows[:, :, :1].contiguous()
    _, S, z = slim.forward(one, one, one, om, 16, "relu")      # one launch
    _, Sg, zg = slim.forward(rows, rows, rows, om, 1, "relu")  # slices of a row, the second one zero
    assert torch.equal(z, zg) and torch.equal(S, Sg)
