"""The network's convolutions and weight gradients at the lattice widths where
their tiles change form: rows of interleaved tiles (64 sites of x and their
ragged neighbours) and the plain ones, one block and several along each axis.
The checks and bounds are those of the layer-by-layer and gradient tests."""

import pytest

import test_gpu_net as N

pytestmark = pytest.mark.gpu

SHAPES = [(8, 8, 64), (8, 16, 56), (8, 24, 120), (16, 8, 72), (8, 8, 136)]


@pytest.mark.parametrize("shape", SHAPES)
def test_layers(shape):
    N.test_each_layer_matches_oracle_on_gpu_inputs(shape)


@pytest.mark.parametrize("shape", SHAPES)
def test_gradients(shape):
    N.test_gradients_match_oracle(shape)
