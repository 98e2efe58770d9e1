"""Restored images against the float64 sum, each pixel within the rounding of
its own terms: single sources at the edges of what reaches an output block,
and models from a few pixels to all of them."""
import numpy as np
import pytest

import oracle
import paper_2501_01461_gb300 as cg

pytestmark = pytest.mark.gpu


def _restore(model, beam, residual=0.0):
    """clean_restore of a given model: a delta PSF at gain 1 moves every
    non-zero pixel of the dirty image into it."""
    import torch
    ny, nx = model.shape
    psf = np.zeros((2 * ny, 2 * nx), np.float32)
    psf[ny, nx] = 1.0
    with cg.Plan(torch.from_numpy(psf).cuda(), ny, nx, gain=1.0,
                 niter=int((model != 0).sum())) as p:
        p.run(torch.from_numpy(model).cuda())
        r, m, _ = p.get()
        out = p.restore(*beam).cpu().numpy()
    assert np.array_equal(m.cpu().numpy(), model) and not r.any()
    return out


def _check(model, bmaj, bmin, pa):
    beam = tuple(float(np.float32(v)) for v in (bmaj, bmin, pa))
    out = _restore(model, beam)
    zero = np.zeros_like(model, dtype=np.float64)
    want = oracle.restore(model, zero, *beam)
    size = oracle.restore(np.abs(model), zero, *beam)
    r = int(5 * bmaj / (2 * np.sqrt(2 * np.log(2))))
    terms = min((2 * r + 1) ** 2, int((model != 0).sum()))
    # a sum of `terms` rounded terms, and each beam value: its argument, up to
    # (r / sigma_minor)^2 / 2, is off by 32 roundings of itself at most (the
    # rotated offset's cancel where the offset is small), expf by a few more
    arg = 0.5 * (r * 2 * np.sqrt(2 * np.log(2)) / bmin) ** 2
    bound = size * 2.0 ** -24 * (terms + 8 + 32 * arg) + 1e-37
    bad = np.abs(out - want) > bound
    assert not bad.any(), (np.argwhere(bad)[:5].tolist(), out[bad][:5], want[bad][:5])


@pytest.mark.parametrize("bmaj,bmin", [(9.5, 7.25), (30.1, 22.0), (1.0, 0.9), (0.4, 0.3)])
def test_sources_at_the_edge_of_a_blocks_reach(bmaj, bmin):
    """Sources whose beams end in, and just before, the output block that
    starts at row 64 and column 64 (or 32 and 32), at its corners and sides."""
    r = int(5 * bmaj / (2 * np.sqrt(2 * np.log(2))))
    model = np.zeros((260, 270), np.float32)
    f = 1.0
    for lo, hi in ((64, 127), (64, 95)):
        for y in (lo - r, lo - r - 1, hi + r, hi + r + 1, 90):
            for x in (lo - r, lo - r - 1, hi + r, hi + r + 1, 100):
                one = np.zeros_like(model)
                one[y, x] = f
                if f == 1.0 or (y, x) in ((lo - r, hi + r), (hi + r, lo - r), (hi + r, 100)):
                    _check(one, bmaj, bmin, 0.6)
                model[y, x] = f
                f *= 0.93
    _check(model, bmaj, bmin, 0.6)


@pytest.mark.parametrize("ny,nx", [(31, 17), (65, 200), (1030, 1040)])
@pytest.mark.parametrize("density", [0.01, 0.15, 0.4, 1.0])
def test_models_of_every_density(ny, nx, density):
    if ny * nx > 1 << 20 and density > 0.15:
        density *= 0.02  # (the float64 sum is a beam a source): see the stripes below
    rng = np.random.default_rng(ny)
    model = np.where(rng.random((ny, nx)) < density, rng.normal(size=(ny, nx)), 0.0)
    _check(np.ascontiguousarray(model, np.float32), 5.5, 4.25, -0.3)


def test_dense_and_empty_parts_side_by_side():
    """Rows that are listed and rows summed whole in the same block, in blocks
    of either size."""
    for ny, nx in ((150, 140), (1030, 1030)):
        rng = np.random.default_rng(7)
        model = np.zeros((ny, nx), np.float32)
        model[40:60, 30:120] = rng.normal(size=(20, 90))
        model[70:130, 100] = rng.normal(size=60)
        model[ny - 3:, nx - 70:] = rng.normal(size=(3, 70))
        _check(model, 14.0, 11.0, 1.2)
