"""Batched tiles on several CTAs: groups that grow while images finish, and
tiles whose only pass a round is shared."""
import numpy as np
import pytest

import paper_2501_01461_gb300 as cg
import synth

pytestmark = pytest.mark.gpu

# (side, tiles, K, niter): the short runs end first, and the longer ones' tiles
# then have more CTAs each
MIXES = [
    [(400, (2, 2), 20, 160), (400, (2, 2), 100, 2400), (512, (1, 1), 30, 900), (256, (1, 1), 0, 500)],
    [(1100, (1, 2), 10, 200)],
    [(600, (2, 2), 5, 60)] * 3 + [(600, (3, 1), 5, 900)],
    [(320, (2, 2), 7, 140)] * 40,
]


@pytest.mark.parametrize("mix", MIXES, ids=lambda m: f"{len(m)}x{m[0][0]}")
def test_batched_groups_equal_solo_runs(mix):
    import torch
    fields = []
    for i, (n, *_) in enumerate(mix[:4]):
        rng = np.random.default_rng(100 * i + n)
        psf = synth.make_psf(2 * n, 2 * n)
        ys, xs, fl = synth.make_sky(n, 25, 0.05, 2.1, rng)
        fields.append((torch.from_numpy(psf).cuda(),
                       torch.from_numpy(synth.make_dirty(psf, n, ys, xs, fl, 1e-3, rng)).cuda()))
    at = [i % len(fields) for i in range(len(mix))]
    kw = [dict(gain=0.1, niter=it, tiles=t, feedback_interval=k) for _, t, k, it in mix]
    with cg.Batch([dict(psf=fields[a][0], ny=m[0], nx=m[0], **q)
                   for a, m, q in zip(at, mix, kw)]) as b:
        b.run([fields[a][1] for a in at], max_rounds=3)
        b.run(None)
        for i in list(range(len(mix)))[:4] + [len(mix) - 1]:
            n = mix[i][0]
            r, m, c = b.get(i)
            with cg.Plan(fields[at[i]][0], n, n, **kw[i]) as p:
                p.run(fields[at[i]][1])
                r0, m0, c0 = p.get()
            assert len(c) == mix[i][3] and np.array_equal(c, c0), i
            assert torch.equal(r, r0) and torch.equal(m, m0), i
