"""The FP32 scan's largest result counts, whose rows are sorted as a whole: a
sort for each full buffer, not for each of the blocks of one slab that the
buffers leave room for."""
import pytest

from test_gpu_merge_runs import _times

pytestmark = pytest.mark.gpu


def test_sorts_of_the_largest_rows():
    """From 400 results to 500 the rows double (512 to 1,024 entries): a sort of
    twice the size, of rows that have room for as many candidates.  1.19 times the
    time; 2.59 with a sort per block."""
    import torch
    some, more = _times(torch, 90, 1000, 16, (400, 500), 1_000_000)
    assert more < 1.8 * some, (some, more)
