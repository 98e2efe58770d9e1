"""Images far from square: the sizes at which launch grids and packed
positions end."""
import numpy as np
import pytest

import oracle
import synth
from gpu_helpers import assert_bit_exact, gpu_clean

pytestmark = pytest.mark.gpu


def test_more_rows_than_a_grids_second_dimension_holds():
    """1,100,000 rows are 68,750 blocks of the plain-load feedback."""
    rng = np.random.default_rng(11)
    dirty, psf = synth.random_image(1_100_000, 3, rng), synth.random_psf(5, 5, rng)
    o = oracle.clean_f32(dirty, psf, 0.1, 6, 0.0)
    assert_bit_exact(gpu_clean(dirty, psf, 0.1, 6, 0.0), o, "1100000 x 3")
