"""The byte counts behind the bench's HBM fractions (no GPU): the single solve and the
batch count the projections' tables by the same rule, at the bytes that a pair takes."""
import inspect

import bench


def test_projector_bytes():
    fwd, bp = bench.projector_bytes(1000, 10, 20, 8)
    assert fwd == 6 * 1000 + 16 * 10 + 24 * 20
    assert bp == 4 * 1000 + 2 * 36 * 8 * 10 + 64 * 10


def test_both_legs_count_by_it():
    for leg in (bench.run_gpu, bench.run_batched):
        source = inspect.getsource(leg)
        assert "projector_bytes(" in source and "* nnz + " not in source
