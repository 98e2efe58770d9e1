"""What plan creation and a PSF change leave behind on their stream."""
import numpy as np
import pytest

import paper_2501_01461_gb300 as cg
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,tiles,K,mode", [(3000, (1, 1), 0, cg.FB_GATHER),
                                            (1024, (2, 2), 10, cg.FB_FFT)])
def test_no_set_up_work_is_left_on_the_plans_stream(n, tiles, K, mode):
    """The PSF's tables (and spectrum) are built when the call that takes the
    PSF returns: a run on another stream may follow at once."""
    import torch
    rng = np.random.default_rng(n)
    psf = torch.from_numpy(synth.make_psf(2 * n, 2 * n)).cuda()
    other = (psf * 2.0).contiguous()
    dirty = torch.from_numpy(synth.random_image(n, n, rng, 1e-2)).cuda()
    kw = dict(gain=0.1, niter=40, tiles=tiles, feedback_interval=K, feedback_mode=mode)
    torch.cuda.synchronize()
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    with cg.Plan(psf, n, n, **kw) as p:
        p.run(dirty)
        want = [v.cpu() for v in p.get()[:2]]
    with cg.Plan(other, n, n, stream=a, **kw) as p:
        assert a.query()
        p.set_psf(psf, stream=a)
        assert a.query()
        p.run(dirty, stream=b)
        got = p.get(stream=b)[:2]
        b.synchronize()
        assert all(torch.equal(g.cpu(), w) for g, w in zip(got, want))
    with cg.Plan(None, n, n, psf_shape=(2 * n, 2 * n), stream=a, **kw) as p:
        p.set_psf_host(psf.cpu().numpy(), stream=b)
        assert b.query()
        p.run(dirty)
        assert all(torch.equal(g.cpu(), w) for g, w in zip(p.get()[:2], want))


def test_results_read_on_another_stream():
    """The component list comes back on the stream it was copied on, behind the
    images (16 MB each) that are on their way there."""
    import torch
    n = 2048
    psf = torch.zeros((2 * n, 2 * n), device="cuda")
    psf[n, n] = 1.0
    dirty = torch.rand((n, n), device="cuda")
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    kw = dict(gain=0.5, niter=500)
    with cg.Plan(psf, n, n, **kw) as p, cg.Batch([dict(psf=psf, ny=n, nx=n, **kw)]) as b:
        p.run(dirty)
        want = p.get()[2]
        assert len(want) == 500
        for _ in range(5):
            assert np.array_equal(p.get(stream=s)[2], want)
        b.run([dirty])
        torch.cuda.synchronize()
        assert np.array_equal(b.get(0, stream=s)[2], want)
