"""Host checks of the workspace sizes (no GPU call): what a query promises to the calls
that run in it."""
import os

import pytest

from paper_2012_11346_gb300 import slim
from paper_2012_11346_gb300 import workloads as W


@pytest.fixture(scope="module", autouse=True)
def built():
    if not os.path.exists(slim._LIB_PATH):
        from paper_2012_11346_gb300 import build
        build.build()


STACKS = [  # d, M, dtype, feature
    (16, 32, "f32", "exp"),
    (32, 112, "f32", "relu"),
    (64, 64, "bf16", "square"),
    (64, 256, "f32", "exp"),
    (128, 256, "bf16", "exp"),
]


@pytest.mark.parametrize("C", [33, 40, 48, 50, 63, 64, 65, 128])
@pytest.mark.parametrize("d,M,dtype,feature", STACKS)
def test_stack_workspace_covers_the_last_slice(d, M, dtype, feature, C):
    """All of a stack's workspace but the segment calls' own follows from the slice length,
    so what a last slice's calls need beyond a full slice's has to be in
    slim_stack_workspace_size."""
    B, H, dt = 1, 2, W.TORCH_DTYPE[dtype]

    def stack(L):
        return slim.stack_workspace_size(B, H, L, d, M, C, 2, dt, feature, True)

    def segment(rows):
        return max(slim.workspace_size(B, H, rows, d, M, rows, dt, feature, b) for b in (False, True))

    for rows in range(1, C):
        assert stack(C + rows) - stack(C) >= segment(rows) - segment(C), rows


# d, M, dtype, feature of the fp32-compute path
PROBLEMS = STACKS + [(64, 128, "f32", "relu"), (128, 160, "bf16", "exp"), (16, 16, "bf16", "square")]


def sizes(B, L, d, M, C, dtype, feature):
    dt = W.TORCH_DTYPE[dtype]
    return tuple(f(B, 1, L, d, M, C, dt, feature, b)
                 for f in (slim.workspace_size, slim.bidir_workspace_size) for b in (False, True))


def rising(values):
    return all(x <= y for a, b in zip(values, values[1:]) for x, y in zip(a, b))


@pytest.mark.parametrize("C", [1, 7, 16, 17, 32, 33, 48, 64, 100, 244, 512, 1024, 5000])
@pytest.mark.parametrize("d,M,dtype,feature", PROBLEMS)
def test_workspace_serves_shorter_sequences_and_fewer_chains(d, M, dtype, feature, C):
    """A buffer for the longest sequence and the most chains serves every other call with the
    same slices, and the size stops growing with L."""
    lengths = sorted({*range(1, 70), *(C * n + r for n in range(1, 12) for r in (0, 1, 33)),
                      300, 1000, 1666, 2155, 3072, 4096, 4608, 8192})
    for B in (1, 3, 48, 64, 512):
        assert rising([sizes(B, L, d, M, C, dtype, feature) for L in lengths])
    for L in (1, 20, 64, 500, 4096, 100000):
        assert rising([sizes(B, L, d, M, C, dtype, feature) for B in range(1, 700, 3)])
    far = max(400 * C, 320 * 64)
    assert sizes(1, far, d, M, C, dtype, feature) == sizes(1, 10 * far, d, M, C, dtype, feature)


@pytest.mark.parametrize("C", [16, 40, 64, 100, 256])
@pytest.mark.parametrize("d,M,dtype,feature", STACKS + [(64, 256, "bf16", "exp"), (64, 128, "bf16", "relu")])
def test_stack_workspace_serves_shorter_sequences(d, M, dtype, feature, C):
    def stack(B, L):
        return tuple(slim.stack_workspace_size(B, 1, L, d, M, C, 2, W.TORCH_DTYPE[dtype], feature, b)
                     for b in (False, True))

    for B in (1, 16, 512):
        assert rising([stack(B, L) for L in (*range(1, C + 70), 2 * C, 7 * C + 5, 40 * C)])
