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


@pytest.mark.parametrize("ny,nx,tiles,K", [
    (3, 32767, (1, 1), 0),      # the longest tile side that selection takes
    (3, 32768, (1, 1), 0),      # the plain loop: a cluster with its rows in shared memory,
    (32800, 2, (1, 2), 10),     # ... two CTAs a tile,
    (33000, 200, (1, 1), 0),    # ... and rows in global memory
    (1, 40000, (1, 1), 0),      # one row: a CTA
])
def test_tiles_around_the_longest_that_selection_takes(ny, nx, tiles, K):
    import torch
    import paper_2501_01461_gb300 as cg
    rng = np.random.default_rng(ny + nx)
    dirty, psf = synth.random_image(ny, nx, rng), synth.random_psf(5, 7, rng)
    niter = 40
    o = oracle.clean_f32(dirty, psf, 0.1, niter, 0.0, tiles, K)
    d_psf, d_dirty = torch.from_numpy(psf).cuda(), torch.from_numpy(dirty).cuda()
    kw = dict(gain=0.1, niter=niter, tiles=tiles, feedback_interval=K)
    with cg.Plan(d_psf, ny, nx, **kw) as p:
        assert p.minor_info()["by_selection"] == (max(ny, nx // tiles[1]) <= 32767)
    assert_bit_exact(gpu_clean(dirty, psf, 0.1, niter, 0.0, tiles, K), o, f"{ny}x{nx}")
    with cg.Batch([dict(psf=d_psf, ny=ny, nx=nx, **kw)]) as b:
        b.run([d_dirty])
        r, m, c = b.get(0)
    assert np.array_equal(c["y"], o.comps["y"]) and np.array_equal(c["x"], o.comps["x"])
    assert np.array_equal(r.cpu().numpy().view(np.uint32), o.residual.view(np.uint32))
    assert np.array_equal(m.cpu().numpy().view(np.uint32), o.model.view(np.uint32))
