"""Plans at the edge of the memory that there is."""
import numpy as np
import pytest

import oracle
import paper_2501_01461_gb300 as cg
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,tiles,K", [(600, (1, 1), 0), (300, (2, 2), 20)])
def test_plan_without_room_for_the_selections_tables(n, tiles, K):
    """A limit that the images, the lists and the beam fit, but not the tables:
    the plan runs the iteration-by-iteration loop, as if there were none."""
    import torch
    rng = np.random.default_rng(n)
    psf = synth.make_psf(2 * n, 2 * n)
    dirty = synth.random_image(n, n, rng, 1e-2)
    niter = 400
    o = oracle.clean_f32(dirty, psf, 0.1, niter, 0.0, tiles, K)
    d_psf, d_dirty = torch.from_numpy(psf).cuda(), torch.from_numpy(dirty).cuda()
    # images, beam table, lists and round buffer; the rest is a few KB
    limit = 8 * n * n + 4 * 129 * 129 + 24 * (niter + 1) + 16 * max(niter, 1) + 40000
    job = dict(psf=d_psf, ny=n, nx=n, gain=0.1, niter=niter, tiles=tiles, feedback_interval=K)
    cg.lib().clean_debug_alloc_limit(limit)
    try:
        p = cg.Plan(d_psf, n, n, gain=0.1, niter=niter, tiles=tiles, feedback_interval=K)
        b = cg.Batch([job])
    finally:
        cg.lib().clean_debug_alloc_limit(-1)
    with cg.Plan(d_psf, n, n, gain=0.1, niter=niter, tiles=tiles, feedback_interval=K) as q:
        assert q.minor_info()["by_selection"]
    assert not p.minor_info()["by_selection"]
    p.run(d_dirty)
    b.run([d_dirty])
    for r, m, c in (p.get(), b.get(0)):
        assert np.array_equal(c["y"], o.comps["y"]) and np.array_equal(c["x"], o.comps["x"])
        assert np.array_equal(r.cpu().numpy().view(np.uint32), o.residual.view(np.uint32))
        assert np.array_equal(m.cpu().numpy().view(np.uint32), o.model.view(np.uint32))
    p.close()
    b.close()
