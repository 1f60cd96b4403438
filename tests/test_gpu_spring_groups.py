"""Mass-spring systems at the edges of how the springs of a step are taken: groups of springs that
do not divide their number (1, 2, 3, 5 and 29 springs), the most springs a system may have (32, so
pairs of masses repeat) with 5 to 8 masses, and with at most 4 masses in a batch large enough for the
wide blocks, whose rest lengths must fit the shared memory.  Same oracle and bars as the pairs' test."""
import itertools

import pytest

import test_gpu_spring_pairs as pairs

pytestmark = pytest.mark.gpu
ms = pairs.ms


@pytest.mark.parametrize("dim,n,count,S", [
    (3, 5, 1, 33), (2, 5, 2, 64), (3, 7, 3, 65), (2, 8, 5, 130), (3, 8, 29, 191), (2, 6, 32, 128), (3, 8, 32, 257),
    (2, 4, 24, 155648), (2, 4, 25, 155648), (3, 4, 32, 155649)])
def test_groups_of_springs_match_oracle(ms, monkeypatch, dim, n, count, S):
    distinct = pairs._springs
    monkeypatch.setattr(pairs, "_springs", lambda n, count, rng: list(
        itertools.islice(itertools.cycle(distinct(n, 28, rng)), count)))
    pairs.test_every_pair_matches_oracle(ms, dim, n, count, S)
