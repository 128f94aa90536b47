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
