"""Results read between launches: the length of a job's component list is
that of the device's state whenever it is asked for, and one allocation holds
a plan's arrays whatever their sizes."""
import numpy as np
import pytest

import paper_2501_01461_gb300 as cg
from paper_2501_01461_gb300 import serve
import synth

pytestmark = pytest.mark.gpu


def _data(ny, nx, seed):
    import torch
    rng = np.random.default_rng(seed)
    m = max(ny, nx)
    psf = synth.make_psf(2 * m, 2 * m)[m - ny:m + ny, m - nx:m + nx]
    dirty = synth.random_image(ny, nx, rng, 1e-2)
    return torch.from_numpy(np.ascontiguousarray(psf)).cuda(), torch.from_numpy(dirty).cuda()


def test_component_counts_follow_the_rounds():
    psf, dirty = _data(96, 96, 1)
    kw = dict(gain=0.1, niter=80, tiles=(2, 2), feedback_interval=5)
    with cg.Batch([dict(psf=psf, ny=96, nx=96, **kw)] * 2) as b:
        for rounds, n in ((0, 0), (1, 20), (2, 60), (-1, 80)):
            b.run([dirty, dirty] if n == 0 else None, max_rounds=rounds)
            assert [len(b.get(i)[2]) for i in (0, 1)] == [n, n]
        b.run([dirty, dirty], max_rounds=1)  # a new run on the same state
        assert len(b.get(1)[2]) == 20
    srv = serve.Server(max_jobs=2)
    try:
        job = serve.Job(psf=psf, dirty=dirty, **kw)
        a = srv.add(job)
        assert len(srv.get(a, (96, 96))[2]) == 0
        srv.step(1)
        c = srv.add(job)
        assert [len(srv.get(j, (96, 96))[2]) for j in (a, c)] == [20, 0]
        srv.step(1)
        assert [len(srv.get(j, (96, 96))[2]) for j in (a, c)] == [40, 20]
    finally:
        srv.close()


@pytest.mark.parametrize("ny,nx,tiles,niter", [(17, 13, (1, 1), 3), (33, 65, (3, 2), 41),
                                               (96, 80, (1, 1), 64)])
def test_arrays_of_odd_sizes_do_not_overlap(ny, nx, tiles, niter):
    """Two plans side by side, run in turn: each gives what it gives alone."""
    psf, dirty = _data(ny, nx, ny)
    kw = dict(gain=0.1, niter=niter, tiles=tiles, feedback_interval=2 if tiles != (1, 1) else 0)
    with cg.Plan(psf, ny, nx, **kw) as p, cg.Plan(psf, ny, nx, **kw) as q:
        p.run(dirty)
        one = p.get()
        q.run(-dirty)
        p.run(dirty)
        two = p.get()
        neg = q.get()
    for a, b, c in zip(one[:2], two[:2], neg[:2]):
        assert np.array_equal(a.cpu().numpy(), b.cpu().numpy())
        assert np.array_equal(a.cpu().numpy(), -c.cpu().numpy())
    assert np.array_equal(one[2], two[2]) and np.array_equal(one[2]["y"], neg[2]["y"])


def test_deep_run_of_a_small_tile():
    """A small tile cleaned far into its noise takes the iteration-by-iteration
    loop; with a threshold that never ends the run, selections."""
    psf, dirty = _data(72, 56, 5)
    out = []
    for thr in (0.0, 1e-30):
        with cg.Plan(psf, 72, 56, gain=0.1, niter=2500, threshold=thr) as p:
            p.run(dirty)
            out.append(p.get())
    (r0, m0, c0), (r1, m1, c1) = out
    assert len(c0) == 2500 and np.array_equal(c0, c1)
    assert np.array_equal(r0.cpu().numpy(), r1.cpu().numpy())
    assert np.array_equal(m0.cpu().numpy(), m1.cpu().numpy())
