"""Which minor loop a plan's rounds launch, with the oracle's bits either way."""
import numpy as np
import pytest

import oracle
import paper_2501_01461_gb300 as cg
import synth
from gpu_helpers import assert_bit_exact

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,tiles,K,want", [
    (128, (1, 1), 1, False), (128, (1, 1), 5, False), (128, (1, 1), 20, True),
    (128, (1, 1), 0, True), (200, (2, 2), 4, False), (200, (2, 2), 16, True),
    (600, (1, 1), 1, True), (600, (1, 1), 3, False), (600, (1, 1), 8, True),
])
def test_short_rounds_take_the_plain_loop(n, tiles, K, want):
    """A selection's start has to be paid for by the round's iterations."""
    import torch
    rng = np.random.default_rng(n + K)
    psf = synth.make_psf(2 * n, 2 * n)
    dirty = synth.random_image(n, n, rng, 1e-2)
    niter = 4 * max(K, 5) * tiles[0] * tiles[1]
    o = oracle.clean_f32(dirty, psf, 0.1, niter, 0.0, tiles, K)
    with cg.Plan(torch.from_numpy(psf).cuda(), n, n, gain=0.1, niter=niter, tiles=tiles,
                 feedback_interval=K) as p:
        assert p.minor_info()["by_selection"] == want
        p.run(torch.from_numpy(dirty).cuda())
        r, m, _ = p.get()
        comps = p.components_with_rounds()
        p.debug_set(cg.DEBUG_MINOR_PATH, 1)
        assert not p.minor_info()["by_selection"]
    assert_bit_exact(dict(residual=r.cpu().numpy(), model=m.cpu().numpy(), comps=comps,
                          n=len(comps["y"])), o, f"{n} {tiles} K {K}")
