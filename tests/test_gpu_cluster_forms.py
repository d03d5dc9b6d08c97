"""The coarse levels' cluster kernel where its forms change: levels of more than
two 4-site groups a thread (one or two sites a row), and first single-block
levels of too many planes for their planes to be pushed to the other blocks
(fetched instead), planes along z and along y.  Check and bounds are those of
the V-cycle's other shapes (against the oracle, and the same bits for 16, 8, 2
and 1 blocks a cluster)."""

import pytest

import test_gpu_march as T

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(90, 90, 2), (70, 180, 1), (2400, 6, 6), (6, 2400, 6), (40, 40, 40)])
def test_vcycle(shape, rng, monkeypatch):
    T.test_fp32_vcycle_matches_oracle_and_itself(shape, rng, monkeypatch)
