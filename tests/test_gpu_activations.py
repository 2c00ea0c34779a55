"""The kernels' sigmoid, tanh and softmax terms over every float: the bits of the
same forms with CUDA's __expf and __fdividef, whose error bounds they therefore
have."""
import pytest

from gpu_common import api

pytestmark = pytest.mark.gpu


def test_every_float_has_the_bits_of_cudas_functions():
    assert api().debug_activations().tolist() == [0, 0, 0]
