"""The selection minor loop (the automatic choice when the caller leaves the
tile groups to the library) against the float32 oracle, bit for bit, at the
sizes where its cells, tables and rounds can go wrong."""
import numpy as np
import pytest

import oracle
import paper_2501_01461_gb300 as cg
import synth
from gpu_helpers import assert_bit_exact, gpu_clean

pytestmark = pytest.mark.gpu


def _field(ny, nx, ps, rng, kind):
    """(dirty, psf): an array PSF (cropped or odd-sized ones off its grid), or
    a random signed one."""
    if kind == "random":
        return synth.random_image(ny, nx, rng), synth.random_psf(*ps, rng)
    big = synth.make_psf(2 * ((max(ps) + 1) // 2) + 2, 2 * ((max(ps) + 1) // 2) + 2)
    c = big.shape[0] // 2
    psf = np.ascontiguousarray(big[c - ps[0] // 2:c - ps[0] // 2 + ps[0],
                                   c - ps[1] // 2:c - ps[1] // 2 + ps[1]])
    dirty = synth.random_image(ny, nx, rng, 1e-3)
    for _ in range(12):
        y, x, f = rng.integers(ny), rng.integers(nx), np.exp(rng.uniform(-3, 0.7))
        y0, x0 = max(0, y - ps[0] // 2), max(0, x - ps[1] // 2)
        sub = psf[y0 - y + ps[0] // 2:, x0 - x + ps[1] // 2:][:ny - y0, :nx - x0]
        dirty[y0:y0 + sub.shape[0], x0:x0 + sub.shape[1]] += np.float32(f) * sub
    return dirty, psf


CASES = [
    # (ny, nx, psf, tiles, K, niter, threshold, trigger, PSF kind)
    (64, 64, (128, 128), (1, 1), 0, 300, 0.0, 0.0, "array"),     # several selections a round
    (65, 63, (131, 127), (1, 1), 0, 65, 0.0, 0.0, "array"),      # cells past the edge, 64 + 1
    (7, 9, (15, 17), (1, 1), 0, 64, 0.0, 0.0, "array"),          # one full and one ragged cell
    (512, 512, (1024, 1024), (1, 1), 0, 200, 0.0, 0.0, "array"),  # 4096 cells: the most kept singly
    (520, 512, (1040, 1024), (1, 1), 0, 200, 0.0, 0.0, "array"),  # the fewest under superblocks
    (1030, 610, (2060, 1220), (1, 1), 0, 150, 0.0, 0.0, "array"),  # ragged superblocks
    (2100, 1100, (2100, 1100), (1, 1), 0, 80, 0.0, 0.0, "array"),  # 8 x 8 cells each, clipped PSF
    (300, 200, (301, 199), (2, 3), 70, 900, 0.0, 0.0, "array"),   # more than one selection a round
    (300, 200, (600, 400), (3, 2), 64, 900, 2e-3, 0.0, "array"),  # exactly one selection a round
    (240, 330, (480, 660), (2, 2), 0, 700, 0.0, 0.4, "array"),    # rounds ended by the flux trigger
    (96, 80, (60, 50), (1, 1), 0, 400, 0.0, 0.0, "random"),       # bounds that reach every cell
    (200, 9, (400, 18), (4, 1), 5, 200, 0.0, 0.0, "random"),
]


@pytest.mark.parametrize("case", CASES, ids=[f"{c[0]}x{c[1]}-t{c[3][0]}x{c[3][1]}-K{c[4]}-{c[8]}"
                                             for c in CASES])
def test_selection_bit_exact(case):
    ny, nx, ps, tiles, K, niter, thr, trigger, kind = case
    rng = np.random.default_rng(ny * 13 + nx)
    dirty, psf = _field(ny, nx, ps, rng, kind)
    o = oracle.clean_f32(dirty, psf, 0.1, niter, thr, tiles, K, trigger=trigger)
    for tma in (0, 1):  # the feedback that subtracts the pending components: automatic, plain
        g = gpu_clean(dirty, psf, 0.1, niter, thr, tiles, K, trigger=trigger, feedback_path=tma)
        assert_bit_exact(g, o, f"{case} feedback {tma}")


def test_selection_of_ties_and_of_values_that_overflow():
    """More equal peaks than candidates (a delta PSF over an integer image),
    and a PSF whose centre makes the residual grow past 1e30: one component a
    pass, as the plain loop does it."""
    rng = np.random.default_rng(3)
    psf = np.zeros((200, 220), np.float32)
    psf[100, 110] = 1.0
    dirty = synth.tie_image(100, 110, rng)
    o = oracle.clean_f32(dirty, psf, 0.5, 150, 0.0, (1, 2), 20)
    assert_bit_exact(gpu_clean(dirty, psf, 0.5, 150, 0.0, (1, 2), 20), o, "ties")
    psf = synth.random_psf(120, 120, rng)
    psf[60, 60] = 1.0
    dirty = synth.random_image(60, 60, rng)
    o = oracle.clean_f32(dirty, psf * np.float32(400.0), 0.1, 20, 0.0)
    assert np.abs(o.residual).max() > 1e30
    assert_bit_exact(gpu_clean(dirty, psf * np.float32(400.0), 0.1, 20, 0.0), o, "growth")


def test_step_leaves_nothing_pending():
    """Between clean_step and clean_feedback the residual holds every
    component of the round on its own tile."""
    import torch
    rng = np.random.default_rng(8)
    dirty, psf = _field(130, 150, (260, 300), rng, "array")
    with cg.Plan(torch.from_numpy(psf).cuda(), 130, 150, gain=0.1, niter=200, tiles=(2, 2),
                 feedback_interval=20) as p:
        p.run(torch.from_numpy(dirty).cuda(), max_rounds=0)
        p.step()
        r, _, _ = p.get()
        o = oracle.clean_f32(dirty, psf, 0.1, 80, 0.0, (2, 2), 0)  # no feedback
        assert np.array_equal(r.cpu().numpy().view(np.uint32), o.residual.view(np.uint32))
        p.feedback()
        p.run(None)
        r, _, _ = p.get()
        o = oracle.clean_f32(dirty, psf, 0.1, 200, 0.0, (2, 2), 20)
        assert np.array_equal(r.cpu().numpy().view(np.uint32), o.residual.view(np.uint32))


@pytest.mark.parametrize("ny,nx,dense", [(64, 64, 0), (65, 200, 0), (31, 17, 1), (130, 70, 1)])
def test_restore_of_sparse_and_dense_models(ny, nx, dense):
    """Output blocks at and past their edges; a model with few and with all
    pixels non-zero (several lists a block), against the float64 restore."""
    import torch
    rng = np.random.default_rng(ny)
    psf = np.zeros((2 * ny, 2 * nx), np.float32)
    psf[ny, nx] = 1.0
    dirty = synth.random_image(ny, nx, rng)
    niter = ny * nx if dense else 20
    with cg.Plan(torch.from_numpy(psf).cuda(), ny, nx, gain=1.0, niter=niter) as p:
        p.run(torch.from_numpy(dirty).cuda())
        r, m, _ = p.get()
        out = p.restore(9.5, 7.25, 0.6).cpu().numpy()
    r, m = r.cpu().numpy(), m.cpu().numpy()
    assert (m != 0).sum() == niter
    want = oracle.restore(m, r, 9.5, 7.25, float(np.float32(0.6)))
    # each of up to 41^2 terms and their sum in float32, beam values to 1e-6
    bound = 41 * 41 * 2.0 ** -24 * np.abs(m).max() * 100 + 2e-6 * np.abs(m).max() * 100
    assert np.abs(out - want).max() <= bound
