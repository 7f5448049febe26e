"""Host-side rules and layouts of the kernels, compiled out of the sources and checked without a GPU."""
import pytest

import csrc_util


def test_weight_only_pair_widths_are_instruction_shapes():
    """The width is the N of a cta_group::2 MMA with M = 256 and A in tensor memory: 32, 64, ... 256."""
    shapes = [(M, N) for M in range(65, 2100, 37) for N in (256, 264, 1024, 4096, 5120, 9480, 11008, 14336, 18944, 32000)]
    widths = csrc_util.wo_pair_widths(shapes)
    assert set(widths) == set(range(64, 257, 32))
