"""The selection groups' bounded waits and the launch counts of a plan."""
import time

import numpy as np
import pytest

import oracle
import paper_2501_01461_gb300 as cg
import synth
from gpu_helpers import assert_bit_exact, gpu_clean

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,tiles,K,niter", [(256, (1, 1), 0, 1000), (256, (2, 2), 20, 400),
                                             (640, (1, 1), 0, 300)])
def test_a_groups_wait_expires_and_poisons(n, tiles, K, niter):
    """Automatic groups: an arrival that never comes ends the run with TIMEOUT in
    bounded time, the plan stays poisoned, and a new one gives the oracle's bits."""
    import torch
    rng = np.random.default_rng(n)
    psf = synth.make_psf(2 * n, 2 * n)
    dirty = synth.random_image(n, n, rng, 1e-2)
    d_psf, d = torch.from_numpy(psf).cuda(), torch.from_numpy(dirty).cuda()
    p = cg.Plan(d_psf, n, n, gain=0.1, niter=niter, tiles=tiles, feedback_interval=K)
    info = p.minor_info()
    assert info["by_selection"] and info["ctas"] > 1
    p.debug_set(cg.DEBUG_SPIN_LIMIT_NS, 20_000_000)
    p.debug_set(cg.DEBUG_FORCE_TIMEOUT, 1)
    t0 = time.time()
    with pytest.raises(cg.CleanError) as e:
        p.run(d)
    assert e.value.status == 5 and time.time() - t0 < 30
    with pytest.raises(cg.CleanError) as e:
        p.run(d)
    assert e.value.status == 5
    p.close()
    o = oracle.clean_f32(dirty, psf, 0.1, niter, 0.0, tiles, K)
    assert_bit_exact(gpu_clean(dirty, psf, 0.1, niter, 0.0, tiles, K), o, "after a timeout")


@pytest.mark.parametrize("n,tables", [(128, 3), (520, 5)])
def test_set_up_launches_are_counted(n, tables):
    """The PSF check, and its tables: two more where cells are kept in blocks."""
    import torch
    with cg.Plan(torch.from_numpy(synth.make_psf(2 * n, 2 * n)).cuda(), n, n, niter=10) as p:
        assert p.stats()["kernel_launches"] == 1 + tables
