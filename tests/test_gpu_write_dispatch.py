"""The write batches of test_gpu_write_batches.py on both sides of the largest
batch that runs as one cluster (2048 keys), over one table and over several."""

import pytest

import test_gpu_write_batches as batches

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2047, 2048, 2049])
@pytest.mark.parametrize("timers", [False, True])
def test_one_table_around_the_largest_cluster_batch(n, timers):
    batches.test_write_batches_match_the_oracle(n, timers)


@pytest.mark.parametrize("n", [2048, 2049])
def test_many_tables_around_the_largest_cluster_batch(n):
    batches.test_write_batches_over_tables_with_and_without_timers(n)
