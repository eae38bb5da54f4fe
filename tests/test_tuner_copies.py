"""How many copies of an LP stand for a batch in the autotuner's trials."""
import pytest


@pytest.mark.parametrize("nnz,batch,copies", [(100, 0, 1), (100, 100, 1), (100, 199, 1), (100, 200, 2), (100, 799, 4), (1 << 20, 1 << 40, 8),
                                              (1 << 30, 1 << 40, 1), (0, 10, 8)])
def test_copies_stand_for_the_batch(nnz, batch, copies):
    from paper_2607_03627_gb300 import tune
    assert tune.copies_of(nnz, batch) == copies
