"""Rounds that the selection hands over to the plain loop (crowded fields deep
in their noise): the same bits, wherever in a round it happens."""
import numpy as np
import pytest

import oracle
import paper_2501_01461_gb300 as cg
import synth
from gpu_helpers import assert_bit_exact

pytestmark = pytest.mark.gpu


def _field(ny, nx, sources, seed, ps=None):
    rng = np.random.default_rng(seed)
    m = max(ny, nx)
    psf = synth.make_psf(2 * m, 2 * m)
    ph, pw = ps or (2 * ny, 2 * nx)
    psf = np.ascontiguousarray(psf[m - ph // 2:m - ph // 2 + ph, m - pw // 2:m - pw // 2 + pw])
    ys, xs, fl = synth.make_sky(m, sources, 0.05, 2.1, rng)
    dirty = synth.make_dirty(synth.make_psf(2 * m, 2 * m), m, ys, xs, fl, 1e-3, rng)[:ny, :nx]
    return np.ascontiguousarray(dirty), psf


def _run(dirty, psf, niter, cycles, **kw):
    import torch
    ny, nx = dirty.shape
    with cg.Plan(torch.from_numpy(psf).cuda(), ny, nx, gain=0.1, niter=niter, **kw) as p:
        if cycles is not None:
            p.debug_set(cg.DEBUG_PLAIN_CYCLES, cycles)
        p.run(torch.from_numpy(dirty).cuda())
        r, m, _ = p.get()
        comps = p.components_with_rounds()
        return dict(residual=r.cpu().numpy(), model=m.cpu().numpy(), comps=comps,
                    n=len(comps["y"])), p.minor_info()


@pytest.mark.parametrize("ny,nx,tiles,K,niter,thr,trigger,kw", [
    (128, 128, (1, 1), 0, 1000, 0.0, 0.0, {}),                 # a cluster takes over
    (77, 130, (1, 1), 0, 900, 2e-3, 0.0, {}),                  # ... until the threshold
    (420, 400, (1, 1), 0, 500, 0.0, 0.0, {}),                  # a grid group
    (128, 96, (1, 1), 0, 600, 0.0, 0.0, dict(mode=cg.UNTILED_GRID)),
    (150, 150, (2, 2), 100, 3000, 0.0, 0.0, {}),               # round after round, in graphs
    (150, 150, (1, 1), 200, 900, 0.0, 0.3, {}),
    (150, 150, (1, 1), 0, 900, 0.0, 0.3, {}),                  # several rounds of one tile
], ids=lambda v: str(v) if isinstance(v, (int, float, tuple)) else None)
def test_handed_over_rounds_equal_the_oracle(ny, nx, tiles, K, niter, thr, trigger, kw):
    dirty, psf = _field(ny, nx, 60, ny + nx)
    o = oracle.clean_f32(dirty, psf, 0.1, niter, thr, tiles, K, trigger=trigger)
    g, info = _run(dirty, psf, niter, 1, threshold=thr, tiles=tiles, feedback_interval=K,
                   feedback_trigger=trigger, **kw)
    assert info["by_selection"] and info["taken_over"] > 0, info
    assert_bit_exact(g, o, "handed over")
    g, info = _run(dirty, psf, niter, 0, threshold=thr, tiles=tiles, feedback_interval=K,
                   feedback_trigger=trigger, **kw)
    assert info["by_selection"] and info["taken_over"] == 0, info
    assert_bit_exact(g, o, "selection alone")


def test_no_hand_over_where_the_plan_has_no_such_launch():
    dirty, psf = _field(64, 64, 5, 1)
    import torch
    for kw in (dict(tiles=(2, 2), feedback_interval=50), dict(feedback_interval=64),
               dict(niter=255)):
        with cg.Plan(torch.from_numpy(psf).cuda(), 64, 64, **{"niter": 2000, **kw}) as p:
            with pytest.raises(cg.CleanError) as e:
                p.debug_set(cg.DEBUG_PLAIN_CYCLES, 1)
            assert e.value.status == 1


def test_crowded_batches_equal_solo_runs():
    """Many small crowded images, one CTA each, and a few with clusters: in a
    batch the rounds go over by themselves."""
    import torch
    for n, side, niter in ((3, 200, 2500), (100, 72, 1500)):
        fields = [_field(side, side, 150, 10 + i) for i in range(min(n, 4))]
        fields = [fields[i % len(fields)] for i in range(n)]
        psfs = [torch.from_numpy(p).cuda() for _, p in fields]
        ds = [torch.from_numpy(d).cuda() for d, _ in fields]
        with cg.Batch([dict(psf=p, ny=side, nx=side, gain=0.1, niter=niter) for p in psfs]) as b:
            b.run(ds)
            for i in range(min(n, 4)):
                d, p = fields[i]
                r, m, c = b.get(i)
                o = oracle.clean_f32(d, p, 0.1, niter, 0.0)
                assert np.array_equal(c["y"], o.comps["y"]) and np.array_equal(c["x"], o.comps["x"])
                assert np.array_equal(r.cpu().numpy().view(np.uint32), o.residual.view(np.uint32))
                assert np.array_equal(m.cpu().numpy().view(np.uint32), o.model.view(np.uint32))


def test_step_of_a_round_that_is_handed_over():
    """clean_step leaves every component of the round on its own tile, also those
    that the plain loop found after the hand-over."""
    import torch
    dirty, psf = _field(150, 150, 60, 3)
    with cg.Plan(torch.from_numpy(psf).cuda(), 150, 150, gain=0.1, niter=1600, tiles=(2, 2),
                 feedback_interval=200) as p:
        p.debug_set(cg.DEBUG_PLAIN_CYCLES, 1)
        p.run(torch.from_numpy(dirty).cuda(), max_rounds=0)
        p.step()
        r = p.get()[0]
        o = oracle.clean_f32(dirty, psf, 0.1, 800, 0.0, (2, 2), 0)  # no feedback
        assert np.array_equal(r.cpu().numpy().view(np.uint32), o.residual.view(np.uint32))
        assert p.minor_info()["taken_over"] == 4
        p.feedback()
        p.run(None)
        r = p.get()[0]
        o = oracle.clean_f32(dirty, psf, 0.1, 1600, 0.0, (2, 2), 200)
        assert np.array_equal(r.cpu().numpy().view(np.uint32), o.residual.view(np.uint32))
